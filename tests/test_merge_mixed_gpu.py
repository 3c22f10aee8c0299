"""The merge of many routers of which few have pending planes, against the
oracle: planes go through the fold, LDCAs that hold bits through the plain OR,
LDCAs known to be zero through neither.
"""
import numpy as np
import pytest

import oracle as O
from test_merge_planes_gpu import BASE, _fill
from test_parity_gpu import assert_same_sketch, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

R = 40                                           # two launches of the plain OR


@pytest.mark.parametrize("k_log2", [6, 8])
@pytest.mark.parametrize("dst_state", ["empty", "planes", "direct", "both"])
@pytest.mark.parametrize("special", [{}, {0: "planes"}, {39: "both"}, {3: "spilled"}, {3: "spilled", 20: "empty", 33: "both"},
                                     {i: "planes" for i in range(1, 39)}, {i: "empty" for i in range(40)}])
def test_few_pending_of_forty(sp, torch, k_log2, dst_state, special):  # noqa: F811
    kw = dict(BASE, k_log2=k_log2, lr=3, lc_log2=6, scan_mode=2, n_routers=R + 1)
    op = oracle_params(kw)
    with sp.SuperPoint(**kw) as ctx:
        states = [special.get(r, "direct") for r in range(R)] + [dst_state]
        osks = [_fill(sp, torch, ctx, O.Sketch(op), r, st, r) for r, st in enumerate(states)]
        union = O.Sketch(op)
        for o in osks:
            union.merge(o)
        for _ in range(2):                       # the sources' planes stay pending: again from the same state
            ctx.merge(list(range(R + 1)), R)
            assert_same_sketch(ctx, union, R)
        for r in (0, 3, 20, 33, 39):
            assert_same_sketch(ctx, osks[r], r)
        sp.sp_reset_range(ctx.ctx, 0, R + 1)
        for r in (3, R):
            seav, ldca = ctx.sketch_image(r)
            assert not seav.any() and not ldca.any(), r
