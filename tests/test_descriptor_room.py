"""The descriptor estimate covers what a plan takes, also where the closed form's displacements do.

A plan gives its bitmaps what the arena holds beside the estimate and 8 MiB of headroom, and runs
in several passes where that is short.  The batch here has 1,500 fields of 961 loads, each in a grid
row of its own: the displacements (16 bytes a load) come to three times the headroom.
"""
import numpy as np
import pytest

from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W

HEADROOM = 8 << 20
N = (64, 256, 256)


def batch(n, shared=False):
    """n candidates of one field each, every one with lists of its own (or all with the same)."""
    star = [W.Access(0, dy, dz, 0) for dy in range(-15, 16) for dz in range(-15, 16)]
    one = W.Config(N=N, B=(32, 1, 1), fields=[W.Field(8, star, strides=W.dense_strides(N))], flops_per_lup=1.0,
                   wave_blocks_override=4)
    cfg, fld, acc = B.marshal([one])
    cfg = np.repeat(cfg, n)
    cfg["wave_blocks_override"] = 1 + np.arange(n) % 7
    if not shared:
        fld = np.repeat(fld, n)
        cfg["field_off"] = np.arange(n)
    return cfg, fld, acc


@pytest.mark.parametrize("shared", [False, True])
def test_estimate_covers_the_lists(shared):
    n = 1500
    plan = B.ws_plan_dry_run(hw=W.a100(), arrays=batch(n, shared))
    assert plan["candidates_ok"] == n
    lists = 16 * (plan["access_entries"] + plan["interval_entries"])
    assert lists == (1 if shared else n) * 2 * 16 * 961         # accesses and displacements
    # the lists, and each candidate's result, key, order and rank
    assert plan["descriptor_bytes"] + HEADROOM >= lists + n * (B.RESULT.itemsize + 16)


def test_estimate_keeps_shared_lists_out():
    """Where the candidates share their lists, nothing is added to the estimate: it grows by the same
    bytes with every seven candidates (their waves repeat), but for the items of the counting, which
    are rounded once a batch (12 bytes each)."""
    d = [B.ws_plan_dry_run(hw=W.a100(), arrays=batch(n, True))["descriptor_bytes"] for n in (70, 140, 1400)]
    assert abs((d[2] - d[1]) - 18 * (d[1] - d[0])) <= 12 * (18 + 1)


@pytest.mark.parametrize("z_extra,entries", [(0, 5 + 1), (1, 5)])
def test_fields_have_runs_or_displacements(z_extra, entries):
    """A 7-point field has displacements of five load rows and one store row in closed form, and five
    merged runs of loads where a walk takes it: planes that are no whole number of rows apart are
    refused."""
    n, dims = 9, (64, 32, 32)
    acc = [W.Access(*o) for o in W.star_offsets(1)] + [W.Access(0, 0, 0, 1)]
    cfgs = [W.Config(N=dims, B=(32, 2, 1), fields=[W.Field(8, acc, strides=(1, 64, 64 * 32 + z_extra))],
                     flops_per_lup=7.0, wave_blocks_override=200) for _ in range(n)]
    plan = B.ws_plan_dry_run(cfgs, W.a100())
    assert plan["candidates_ok"] == n and plan["interval_entries"] == n * entries
    for walk in (B.WS_WALK_SEGMENT, B.WS_WALK_ADDRESS):
        assert B.ws_plan_dry_run(cfgs, W.a100(), tuning={"walk": walk})["interval_entries"] == n * (5 if z_extra else 11)


def test_candidates_of_one_field_keep_their_own_kind_of_list():
    """Blocks of four points are shorter than a reach of four and take the row walk, blocks of 32 do not:
    the field's list without runs and the one with them and their covers are shared apart."""
    one, dims = [], (128, 64, 64)
    star = [W.Access(*o) for o in W.star_offsets(4)] + [W.Access(0, 0, 0, 1)]
    fields = [W.Field(8, star, strides=W.dense_strides(dims))]
    for block in ((32, 4, 1), (4, 8, 4), (64, 2, 1), (4, 4, 8)):
        one.append(W.Config(N=dims, B=block, fields=fields, flops_per_lup=25.0))
    runs, dsp = 17, 17 + 1
    want = {(32,): dsp, (4,): runs + dsp}
    for keep in ((32,), (4,), (32, 4)):
        cfgs = [c for c in one if (c.B[0] == 4) == (4 in keep) or len(keep) == 2]
        plan = B.ws_plan_dry_run(cfgs, W.a100())
        assert plan["interval_entries"] == (want[keep] if len(keep) == 1 else sum(want.values())), keep


@pytest.mark.gpu
def test_small_arena_runs_in_passes():
    """The arena holds descriptors and some of the bitmaps: results as in one with room for all."""
    arrays = batch(1500)
    want = None
    for arena in (1 << 30, 104 << 20):
        ctx = B.Context(0, arena)
        try:
            with B.Plan(ctx, hw=W.a100(), arrays=arrays) as p:
                passes = p.profile()["passes"]
                p.execute(B.WS_MODE_BATCHED)
                res, order = p.results()
        finally:
            ctx.close()
        assert (res["status"] == 0).all()
        if want is None:
            want = (res.tobytes(), order.tobytes())
        assert passes == 1 if arena == 1 << 30 else passes > 1
        assert (res.tobytes(), order.tobytes()) == want
