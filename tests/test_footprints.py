"""Closed-form footprints (row by row, without bitmaps) against the oracle and the address walk.

Counts are whole numbers and have to agree exactly, and the results of the closed form and of the
per-address walk bit for bit.  The layouts sit on the edges of the closed form's rule: rows dense
and padded, planes that join without a row to spare, planes of one row, one plane only, negative
and shared alignments, rests that reach over a row's end, waves that leave a gap between the end
of one block row and the start of the next, spans beyond 2^31 and 2^32 bytes, z sets moved by any
number of bytes, fields that are copies of one another moved by whole lines or by less, folds cut
by the domain's end, and layouts the rule refuses (x strides beyond a sector, descending rows),
which the walks count beside them.
"""
import os

import pytest

import oracle
from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W


def layouts(rng, N, esize):
    """Strides: dense, padded rows, padded planes, one row of slack, wide spans, refused ones."""
    kind = rng.randint(0, 9)
    px = N[0] + rng.choice((0, 0, 1, 5, 32 - N[0] % 32))
    if kind <= 3:
        return (1, px, px * N[1])
    if kind == 4:
        return (1, px, px * (N[1] + rng.choice((1, 2, 9))))
    if kind == 5:                                    # x steps of more than one element, up to a sector
        sx = max(1, 32 // esize)
        return (sx, sx * px, sx * px * N[1])
    if kind == 6:                                    # rows far apart: a span beyond 2^31 bytes, or beyond 2^32
        return (1, ((1 << 22) + rng.choice((0, 24, 1))) // esize, ((1 << 22) // esize) * rng.choice((N[1], N[1] + 3)))
    if kind == 7:                                    # planes no whole number of rows apart
        return (1, px, px * N[1] + rng.randint(1, max(1, px - 1)))
    if kind == 8:                                    # refused: beyond a sector a point
        return (64 // esize + 1, (64 // esize + 1) * px, (64 // esize + 1) * px * N[1])
    return (1, -px, px * N[1] * 2)                   # refused: descending rows


def candidates(seed, n):
    rng = W.SplitMix64(seed)
    out = []
    for _ in range(n):
        axis, fold = rng.choice([(0, 1), (0, 1), (1, 2), (2, 4), (1, 4), (2, 3)])
        block = rng.choice([(32, 2, 1), (8, 4, 2), (5, 3, 3), (4, 8, 1), (64, 1, 2), (1, 8, 4), (16, 1, 8), (33, 1, 1)])
        N = (rng.randint(1, 90), rng.choice((1, 2, 7, 16, 25)), rng.choice((1, 2, 9, 16, 40)))
        esize = rng.choice((1, 2, 4, 8, 16))
        st = layouts(rng, N, esize)
        if abs(st[1]) * esize > 1 << 21:
            N = (N[0], min(N[1], 16), min(N[2], 70))
        r, base = rng.choice((0, 1, 2, 4)), rng.randint(-130, 130)
        kind = rng.randint(0, 3)
        fields = []
        for k in range(rng.choice((1, 1, 2, 3, 7))):
            if kind == 0:                            # star
                accs = {W.Access(d * (a == 0), d * (a == 1), d * (a == 2), 0, 0) for a in range(3) for d in range(-r, r + 1)}
            elif kind == 1:                          # a few of a box, not the same in every field
                accs = {W.Access(rng.randint(-r, r), rng.randint(-r, r), rng.randint(-r, r), 0, 0) for _ in range(6)}
            elif kind == 2:                          # one offset: copies moved by a line or by less
                accs = {W.Access(k % 2, 0, 0, 0, 0)}
            else:                                    # rests of up to a row
                accs = {W.Access(rng.choice((-N[0] // 2, 0, N[0] // 2)), rng.randint(-1, 1), 0, 0, 0) for _ in range(3)}
            if rng.randint(0, 2):
                accs.add(W.Access(0, 0, 0, 1, 0))
                if rng.randint(0, 2) == 0:
                    accs.add(W.Access(rng.randint(-1, 1), 1, 0, 1, 0))
            fields.append(W.Field(esize, sorted(accs, key=lambda a: (a.dx, a.dy, a.dz, a.is_store, a.dc)),
                                  align=base + k * rng.choice((0, 128, 4096, 32, 7)), strides=st))
        out.append(W.Config(N=N, B=block, fields=fields, fold_axis=axis, fold=fold, flops_per_lup=2.0,
                            wave_blocks_override=rng.choice((0, 1, 2, 3, 5, 9, 14)), address_mode=rng.randint(0, 5) == 0))
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("seed", [31, 32, 33, 34])
def test_footprints_match_oracle_and_address_walk(seed):
    hw = W.Hardware(sms=3, max_blocks_sm=4)
    cfgs = candidates(seed, 200)
    want = oracle.estimate(cfgs, hw, threads=len(os.sched_getaffinity(0)))
    ctx, out = B.Context(0, 24 << 30), []
    try:
        for walk in (B.WS_WALK_INTERVAL, B.WS_WALK_ADDRESS):
            with B.Plan(ctx, cfgs, hw, tuning={"walk": walk}) as p:
                for mode in (B.WS_MODE_BATCHED, B.WS_MODE_PLAIN):
                    p.execute(mode)
                    res, order = p.results()
                    out.append((res.tobytes(), order.tobytes()))
                    assert out[-1] == out[0], (walk, mode)
    finally:
        ctx.close()
    for i, (got, w) in enumerate(zip(B.results_to_dicts(res), want)):
        assert got["status"] == w["status"], i
        if w["status"] == 0:
            for k in B.RESULT_INT:
                assert got[k] == w[k], (i, k, got[k], w[k])


@pytest.mark.gpu
@pytest.mark.parametrize("B0,r,walked", [(8, 4, False), (16, 1, False), (4, 2, False), (4, 4, True)])
def test_closed_form_leaves_no_rows_to_walk(B0, r, walked):
    """Stars are counted without a bitmap, but for the block where its runs of four points are
    shorter than a reach of four spreads its offsets."""
    star = {W.Access(d * (a == 0), d * (a == 1), d * (a == 2), 0, 0) for a in range(3) for d in range(-r, r + 1)}
    cfg = W.Config(N=(96, 40, 40), B=(B0, 4, 2), flops_per_lup=1.0,
                   fields=[W.Field(8, sorted(star, key=lambda a: (a.dx, a.dy, a.dz)), strides=(1, 96, 96 * 40))])
    ctx = B.Context(0, 1 << 30)
    try:
        with B.Plan(ctx, [cfg], W.a100()) as p:
            prof = p.profile()
    finally:
        ctx.close()
    assert (prof["row_reds"] > 0) == walked and (prof["count_bytes"] > 0) == walked
