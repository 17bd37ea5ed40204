"""Where the closed form of the footprints ends: 2^32 sectors, and row numbers of 32 bits.

A closed-form item sums its counts in 32 bits, so a field whose wave may hold 2^32 sectors or more
takes the address walk.  The arrays of those tests are dense and aligned, one element a sector, and
their waves cover the whole domain: the counts follow from the number of points alone.

Target rows are numbered in 32 bits, too, up to two planes behind the last one: where planes lie
so far apart that these numbers do not fit, the address walk is taken.
"""
import pytest

import oracle
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


def far(N, row, q):
    """Loads of 8-byte elements in rows of 256 bytes, q rows a plane, `row` rows from the point."""
    return W.Config(N=N, B=(8, 2, 1), fields=[W.Field(8, [W.Access(0, 0, 0, 0, 32 * row)], strides=(1, 32, 32 * q))],
                    flops_per_lup=1.0, wave_blocks_override=1 << 20)


FAR_Q = (1 << 30) - (1 << 21)
FAR = [
    (far((32, 4, 2), 5, FAR_Q // 2), True),
    (far((32, 4, 2), (1 << 28) - 2, 1 << 28), True),
    (far((32, 4, 1), (1 << 28) - 2, FAR_Q), True),           # one plane: the rows to the next do not matter
    (far((32, 4, 2), 5, FAR_Q), False),
    (far((32, 4, 2), (1 << 28) - 2, FAR_Q), False),          # target rows 2^28 - 2 .. and two planes from there
    (far((32, 4, 2), 2 - (1 << 28), FAR_Q), False),
]


@pytest.mark.parametrize("cfg,closed", FAR)
def test_far_rows_leave_the_closed_form(cfg, closed):
    plan = B.ws_plan_dry_run([cfg], W.a100())
    assert plan["candidates_ok"] == 1
    assert (plan["row_items"] > 0) == closed


@pytest.mark.gpu
def test_far_rows_match_oracle():
    cfgs = [c for c, _ in FAR]
    want = oracle.estimate(cfgs, W.a100())
    ctx = B.Context(0, 12 << 30)
    try:
        res, _ = B.ws_estimate_batch(ctx, cfgs, W.a100())
    finally:
        ctx.close()
    for i, (got, w) in enumerate(zip(B.results_to_dicts(res), want)):
        assert got["status"] == w["status"] == B.WS_OK
        for k in B.RESULT_INT:
            assert got[k] == w[k], (i, k, got[k], w[k])
