"""Batched binned scans of streams whose sizes are whole tiles or a pair off,
starting on a 16-byte boundary or 8 bytes past one, against the oracle.
"""
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_sketch, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

KW = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), k_log2=8, lr=3, lc_log2=9, theta=64, seed=171, scan_mode=2)


@pytest.mark.parametrize("shape", [0, 2])                       # tiles of 8,192 and of 4,096 pairs
@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("sizes", [[8192] * 130, [16384, 8191, 8192, 8193, 1], [4096, 12288, 4097, 2], [8192 * 152], [8192 * 152 + 1],
                                   [4096 * 304 - 1]])
def test_whole_tiles(sp, torch, sizes, offset, shape):  # noqa: F811
    parts = [W.uniform_pairs(n, seed=1700 + i, n_hosts=max(1, n // 20)) for i, n in enumerate(sizes)]
    tens = [dev(torch, p, offset) for p in parts]
    osk = O.Sketch(oracle_params(KW))
    for p in parts:
        osk.update(p)
    with sp.SuperPoint(**KW) as ctx:
        sp.sp_set_binned_shape(ctx.ctx, shape)
        sp.sp_update_batched(ctx.ctx, [0] * len(tens), tens)
        assert_same_sketch(ctx, osk)
