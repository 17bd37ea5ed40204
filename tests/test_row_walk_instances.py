"""Passes of row-walk items alone, of both kinds together, and of both apart.

The row walk has a kernel of its own (four CTAs an SM) for passes without closed-form items and for
those in which it outweighs them; otherwise the closed form's kernel takes both.  Descending rows are
refused by the closed form, everything else here is taken by it.
"""
import dataclasses
import os

import pytest

import oracle
from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def descending(cfgs):
    """The same candidates with rows of descending addresses (shared field lists stay shared)."""
    memo = {}
    for c in cfgs:
        if id(c.fields) not in memo:
            memo[id(c.fields)] = [dataclasses.replace(f, strides=(f.strides[0], -f.strides[1], f.strides[2]))
                                  for f in c.fields]
    return [dataclasses.replace(c, fields=memo[id(c.fields)]) for c in cfgs]


def run(cfgs, hw, walk, arena=6 << 30):
    ctx, out = B.Context(0, arena), []
    try:
        with B.Plan(ctx, cfgs, hw, tuning={"walk": walk}) as p:
            launches = p.profile()["launches"]
            for mode in (B.WS_MODE_BATCHED, B.WS_MODE_PLAIN):
                p.execute(mode)
                res, order = p.results()
                out.append((res.tobytes(), order.tobytes()))
    finally:
        ctx.close()
    assert out[0] == out[1]
    return res, out[0], launches


def test_row_walk_alone_matches_oracle():
    hw = W.Hardware(sms=3, max_blocks_sm=2)
    cfgs = descending(W.stencil_25pt_sweep(N=(48, 37, 29))[::12])
    cfgs += descending([c for c in W.lbm_sweep(N=(40, 33, 18))[::40]])
    want = oracle.estimate(cfgs, hw, threads=len(os.sched_getaffinity(0)))
    res, got, launches = run(cfgs, hw, B.WS_WALK_INTERVAL)
    assert launches == 6 and got == run(cfgs, hw, B.WS_WALK_ADDRESS)[1]
    for i, (r, w) in enumerate(zip(B.results_to_dicts(res), want)):
        assert r["status"] == w["status"] == 0
        for k in B.RESULT_INT:
            assert r[k] == w[k], (i, k, r[k], w[k])


@pytest.mark.parametrize("refused,closed,launches", [(84, 0, 6), (84, 1, 7), (84, 16, 7), (8, 84, 6), (1, 1, 6)])
def test_row_walk_beside_the_closed_form(refused, closed, launches):
    """Together (one launch of the footprints) where the closed form is the larger part or the row
    walk is small, apart (two) where the row walk outweighs it."""
    sweep = W.lbm_sweep(N=(256, 256, 256))[::9]
    cfgs = descending(sweep)[:refused] + sweep[:closed]
    res, got, n = run(cfgs, W.a100(), B.WS_WALK_INTERVAL)
    assert n == launches and (res["status"] == 0).all()
    assert got == run(cfgs, W.a100(), B.WS_WALK_SEGMENT)[1]
