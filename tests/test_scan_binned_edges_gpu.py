"""The binned scan at the edges of its tiles, against the oracle: whole tiles
and small ones (one block's, one round over the blocks, a pair more or less),
streams that start 8 bytes off a 16-byte boundary, odd pairs at either end,
lists of a few hips, planes of every row split, and many streams per launch.
"""
import numpy as np
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_sketch, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

ROUND = 152 * 8192                    # a round of whole tiles on a GB300
KW = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), theta=16, seed=81, scan_mode=2)


@pytest.mark.parametrize("shape", [0, 2])
@pytest.mark.parametrize("n,off", [(1, 1), (2, 1), (3, 1), (65, 0), (8191, 1), (8193, 0), (ROUND - 1, 0), (ROUND, 0),
                                   (ROUND, 1), (ROUND + 1, 0), (ROUND + 2, 1), (2 * ROUND + 64 * 152 + 3, 1)])
def test_sizes_around_a_round(sp, torch, n, off, shape):  # noqa: F811
    kw = dict(KW, k_log2=9, lr=2, lc_log2=9)
    x = W.uniform_pairs(n, seed=n % 1000 + 1, n_hosts=max(1, n // 30))
    with sp.SuperPoint(**kw) as ctx:
        sp.sp_set_binned_shape(ctx.ctx, shape)
        ctx.update(dev(torch, x, off))
        osk = O.Sketch(oracle_params(kw)).update(x)
        assert_same_sketch(ctx, osk)
        more = W.uniform_pairs(777, seed=5)                   # on pending planes
        ctx.update(dev(torch, more, 1 - off))
        ctx.update(dev(torch, more, off))
        assert_same_sketch(ctx, osk.update(more))


@pytest.mark.parametrize("k_log2,lr,lc_log2", [(5, 1, 5), (6, 3, 5), (10, 8, 11), (10, 4, 14), (10, 4, 16), (8, 4, 18)])
def test_plane_shapes(sp, torch, k_log2, lr, lc_log2):  # noqa: F811
    kw = dict(KW, k_log2=k_log2, lr=lr, lc_log2=lc_log2)
    x = W.uniform_pairs(300007, seed=lr, n_hosts=9000)
    with sp.SuperPoint(**kw) as ctx:
        for shape in (0, 1):
            sp.sp_reset(ctx.ctx, 0)
            sp.sp_set_binned_shape(ctx.ctx, shape)
            ctx.update(dev(torch, x[:200001], 1))
            ctx.update(dev(torch, x[200001:]))
            assert_same_sketch(ctx, O.Sketch(oracle_params(kw)).update(x))


def test_many_odd_streams_in_a_launch(sp, torch):  # noqa: F811
    """300 streams of 0 to 9,000 pairs, half of them misaligned, in appending
    launches of up to 128."""
    kw = dict(KW, k_log2=10, lr=4, lc_log2=10)
    rng = np.random.default_rng(83)
    parts = [W.uniform_pairs(int(n), seed=8300 + i, n_hosts=500)
             for i, n in enumerate(np.concatenate([np.arange(40), rng.integers(0, 9000, 260)]))]
    with sp.SuperPoint(**kw) as ctx:
        sp.sp_update_batched(ctx.ctx, [0] * len(parts), [dev(torch, p, i & 1) for i, p in enumerate(parts)])
        assert_same_sketch(ctx, O.Sketch(oracle_params(kw)).update(np.concatenate(parts)))


@pytest.mark.parametrize("shape", [0, 2])
@pytest.mark.parametrize("peers", [2, 300, 500, 700])
def test_rows_that_overflow(sp, torch, peers, shape):  # noqa: F811
    """Few distinct peers crowd few bins: rows overflow now and then (the pairs
    wait for the end of the round) or all the time (L2 REDs)."""
    kw = dict(KW, k_log2=10, lr=4, lc_log2=12, theta=8, n_routers=2)
    rng = np.random.default_rng(peers)
    n = 2 * ROUND + 12345
    oips = rng.integers(0, 2**32, peers, dtype=np.uint32)
    x = np.stack([rng.integers(0, 2**32, n, dtype=np.uint32), oips[rng.integers(0, peers, n)]], 1)
    with sp.SuperPoint(**kw) as ctx:
        sp.sp_set_binned_shape(ctx.ctx, shape)
        ctx.update(dev(torch, x))
        osk = O.Sketch(oracle_params(kw)).update(x)
        ctx.merge([0], 1)
        assert_same_sketch(ctx, osk, 1)
        assert_same_sketch(ctx, osk, 0)
        ctx.reset(0)
        seav, ldca = ctx.sketch_image(0)
        assert not seav.any() and not ldca.any()
