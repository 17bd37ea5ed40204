"""Per-instruction counts of the representative block by access codes, against the oracle.

Where the block's footprints are made elsewhere, the enumeration counts distinct sectors and bank
cycles once per code: the place of an access in the period of sectors and banks, and the first
folded point that needs it where some thread of the block has fewer points than the fold.  The
counts are whole numbers and have to agree exactly.  The candidates sit on the edges of that rule:
blocks cut by the domain's end along the folding axis, loads and stores with one code, fields
that differ by a period or by a byte, more fields than a group takes, periods from one sector to
the largest, and (64 banks of 16 bytes folded by 4) more codes than the list has room for.
"""
import os

import pytest

import oracle
from paper_2204_14242_gb300 import binding as B
from paper_2204_14242_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def candidates(seed, n):
    rng = W.SplitMix64(seed)
    out = []
    for _ in range(n):
        axis, fold = rng.choice([(0, 1), (1, 2), (2, 4), (1, 4), (2, 3)])
        block = rng.choice([(32, 2, 1), (8, 4, 2), (5, 3, 3), (64, 1, 2), (4, 8, 4), (33, 1, 1)])
        N = (rng.randint(3, 90), rng.randint(1, 30), rng.randint(1, 30))
        esize = rng.choice((1, 4, 8, 16))
        px = N[0] + rng.choice((0, 1, 7, 32 - N[0] % 32))
        st = (1, px, px * (N[1] + rng.randint(0, 2)))
        base = rng.randint(-70, 70)
        fields = []
        for k in range(rng.choice((1, 2, 5, 19))):
            accs = {W.Access(rng.randint(-3, 3), rng.randint(-3, 3), rng.randint(-3, 3), 0, 0)
                    for _ in range(rng.randint(0, 12))}
            if rng.randint(0, 1) or not accs:
                accs.add(W.Access(0, 0, 0, 1, 0))
                accs.add(W.Access(rng.randint(-1, 1), rng.randint(-1, 1), 0, 1, 0))
            fields.append(W.Field(esize, sorted(accs, key=lambda a: (a.dx, a.dy, a.dz, a.is_store, a.dc)),
                                  align=base + rng.choice((0, 128, 1024, 1, esize)) * k, strides=st))
        out.append(W.Config(N=N, B=block, fields=fields, fold_axis=axis, fold=fold,
                            wave_blocks_override=rng.choice((0, 1, 2, 5)), flops_per_lup=2.0))
    return out


@pytest.mark.parametrize("banks,bank_bytes,pair", [(16, 8, 1024), (32, 4, 512), (2, 4, 64), (64, 16, 1024)])
def test_block_counts_by_access_codes(banks, bank_bytes, pair):
    hw = W.Hardware(sms=3, max_blocks_sm=2, banks=banks, bank_bytes=bank_bytes, pair_dist_bytes=pair)
    cfgs = candidates(banks + bank_bytes + pair, 160)
    want = oracle.estimate(cfgs, hw, threads=len(os.sched_getaffinity(0)))
    ctx = B.Context(0, 4 << 30)
    try:
        res, _ = B.ws_estimate_batch(ctx, cfgs, hw)
    finally:
        ctx.close()
    for i, (got, w) in enumerate(zip(B.results_to_dicts(res), want)):
        assert got["status"] == w["status"], i
        if w["status"] == 0:
            for k in B.RESULT_INT:
                assert got[k] == w[k], (i, k, got[k], w[k])
