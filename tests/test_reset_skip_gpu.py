"""Resets large enough to skip LDCAs that are known to be zero: routers in every
state, ranges that are no multiple of 32 and start anywhere, and one router.
"""
import pytest

import oracle as O
from test_merge_planes_gpu import _fill
from test_parity_gpu import assert_same_sketch, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

STATES = ["planes", "empty", "spilled", "direct", "both"]


@pytest.mark.parametrize("routers,first,count,lc_log2", [(40, 3, 36, 12), (70, 0, 70, 12), (33, 1, 32, 12), (2, 1, 1, 16),
                                                         (2, 0, 2, 16)])
def test_ranges(sp, torch, routers, first, count, lc_log2):  # noqa: F811
    kw = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), theta=64, seed=71, k_log2=10, lr=4, lc_log2=lc_log2, scan_mode=2,
              n_routers=routers)
    op = oracle_params(kw)
    with sp.SuperPoint(**kw) as ctx:
        image = torch.empty(sp.sp_copy_sketch_bytes(ctx.ctx), dtype=torch.uint8, device="cuda")
        for step in range(5):
            osks = {}
            for i in range(step % 2, routers, 7):            # few routers are touched, each in another state
                osks[i] = _fill(sp, torch, ctx, O.Sketch(op), i, STATES[(i + step) % 5], i % 3)
            sp.sp_reset_range(ctx.ctx, first, count)
            for r in range(routers):
                if first <= r < first + count:
                    sp.sp_copy_sketch(ctx.ctx, r, image)
                    assert not image.any(), (step, r)
                elif r in osks:
                    assert_same_sketch(ctx, osks[r], r)
            sp.sp_reset_range(ctx.ctx, 0, routers)
