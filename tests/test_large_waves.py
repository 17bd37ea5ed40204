"""Waves of many row slots: what the closed form does not count is shared out by their number.

A slot is one thread row of one block row; in a batch of fewer than 2.4 million of them an item takes
at most 256.
"""
import pytest

from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W

SLOTS = 256


def star(N, block, wave, esize=8, fold_axis=0, fold=1):
    return W.Config(N=N, B=block, fields=W.copy_fields(N, W.star_offsets(1), esize=esize), flops_per_lup=7.0,
                    wave_blocks_override=wave, fold_axis=fold_axis, fold=fold)


@pytest.mark.parametrize("wave", [64, 4096, 400000])
@pytest.mark.parametrize("others", [0, 3000])
def test_items_follow_the_wave(wave, others):
    """400,000 blocks of 4 x 8 x 4 are 3125 block rows of 128 blocks, 32 thread rows each."""
    cfg = star((512, 512, 512), (4, 8, 4), wave)
    small = [star((64, 16, 16), (32, 2, 1), 4)] * others
    base = B.ws_plan_dry_run(small, W.a100())["row_items"] if others else 0
    plan = B.ws_plan_dry_run(small + [cfg], W.a100())
    assert plan["row_items"] - base >= -(-wave // 128) * 32 // SLOTS


@pytest.mark.gpu
@pytest.mark.parametrize("block,waves", [
    ((4, 8, 4), (1, 1023, 1024, 1025, 8193, 1 << 20)),      # 16 blocks a block row: 1024 blocks are 2048 slots
    ((3, 5, 7), (1, 700, 5000, 1 << 20)),                   # odd blocks, up to the whole domain
    ((64, 1, 1), (127, 128, 8192, 8193, 16385, 1 << 20))])
def test_large_waves_match_the_address_walk(block, waves):
    N = (64, 131, 250)
    cfgs = [star(N, block, w, esize, axis, fold) for w in waves for esize in (4, 8)
            for axis, fold in ((0, 1), (1, 3), (2, 2))]
    ctx, out = B.Context(0, 4 << 30), []
    try:
        for walk in (B.WS_WALK_INTERVAL, B.WS_WALK_ADDRESS):
            with B.Plan(ctx, cfgs, W.a100(), tuning={"walk": walk}) as p:
                for mode in (B.WS_MODE_BATCHED, B.WS_MODE_PLAIN):
                    p.execute(mode)
                    res, order = p.results()
                    out.append((res.tobytes(), order.tobytes()))
    finally:
        ctx.close()
    assert (res["status"] == 0).all()
    assert all(o == out[0] for o in out)
