"""The merge of routers whose binned planes are still pending, and the reset
that skips an LDCA known to be zero, against the oracle.

Sources and destination take every state a router can be in: empty, direct
bits in the LDCA, pending planes, both, and planes beside bits that spilled
past full lists.  k = 64 takes k_fold, k >= 256 k_fold8; 40 sources take two
launches.
"""
import numpy as np
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_sketch, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

BASE = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), theta=64, seed=71)
# (k_log2, lr, lc_log2): W = lr 2^lc / 32 plane words, not always a multiple of 8
SHAPES = [(6, 3, 7), (7, 2, 5), (8, 3, 6), (10, 4, 10), (9, 1, 5)]


def _pairs(state, i):
    if state == "spilled":                       # one oip: a single bin, rows and lists overflow
        rng = np.random.default_rng(710 + i)
        return np.stack([rng.integers(0, 2**32, 30000, dtype=np.uint32), np.full(30000, 7, np.uint32)], 1)
    return W.uniform_pairs(4001 + 17 * i, seed=700 + i, n_hosts=300)


def _fill(sp, torch, ctx, osk, router, state, i):  # noqa: F811
    if state in ("direct", "both"):              # an image ORed in: bits straight in the LDCA
        x = _pairs("direct", i + 50)
        with sp.SuperPoint(**dict(BASE, k_log2=ctx.params.k_log2, lr=ctx.params.lr, lc_log2=ctx.params.lc_log2)) as one:
            one.update(dev(torch, x))            # a small update: direct
            img = torch.zeros(sp.sp_copy_sketch_bytes(one.ctx), dtype=torch.uint8, device="cuda")
            sp.sp_copy_sketch(one.ctx, 0, img)
            sp.sp_merge_device(ctx.ctx, [img], router)
            torch.cuda.synchronize()
        osk.update(x)
    if state in ("planes", "both", "spilled"):
        x = _pairs(state, i)
        ctx.update(dev(torch, x), router=router)
        osk.update(x)
    return osk


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dst_state", ["empty", "direct", "planes", "both", "spilled"])
def test_merge_of_every_state(sp, torch, shape, dst_state):  # noqa: F811
    kw = dict(BASE, k_log2=shape[0], lr=shape[1], lc_log2=shape[2], scan_mode=2, n_routers=6)
    op = oracle_params(kw)
    states = ["planes", "empty", "spilled", "direct", "both", dst_state]
    with sp.SuperPoint(**kw) as ctx:
        for step in range(2):                    # the second pass follows a reset of routers in every state
            osks = [_fill(sp, torch, ctx, O.Sketch(op), r, st, 10 * r + step) for r, st in enumerate(states)]
            ctx.merge([0, 1, 2, 3, 4, 5], 5)
            union = O.Sketch(op)
            for o in osks:
                union.merge(o)
            got, n, _ = ctx.detect(router=5, threshold=64)
            want, n_want, _ = union.detect(64)
            assert n == n_want and np.array_equal(got, want)
            assert_same_sketch(ctx, union, 5)
            extra = _pairs("planes", 90 + step)  # the sources go on after the merge
            ctx.update(dev(torch, extra), router=0)
            osks[0].update(extra)
            for r in range(5):
                assert_same_sketch(ctx, osks[r], r)
            sp.sp_reset_range(ctx.ctx, 0, 6)
            if step:
                for r in range(6):
                    seav, ldca = ctx.sketch_image(r)
                    assert not seav.any() and not ldca.any(), r


@pytest.mark.parametrize("k_log2", [6, 8])
def test_merge_of_forty_pending_routers(sp, torch, k_log2):  # noqa: F811
    kw = dict(BASE, k_log2=k_log2, lr=3, lc_log2=6, scan_mode=2, n_routers=41)
    osk = O.Sketch(oracle_params(kw))
    with sp.SuperPoint(**kw) as ctx:
        for step in range(2):
            osk = O.Sketch(oracle_params(kw))
            for r in range(40):
                x = _pairs("spilled" if r == 35 else "planes", 100 * step + r)
                ctx.update(dev(torch, x), router=r)
                osk.update(x)
            ctx.merge(list(range(40)), 40)
            assert_same_sketch(ctx, osk, 40)
            sp.sp_reset_range(ctx.ctx, 0, 41)    # sources never folded: their LDCAs are skipped but 35's


def test_reset_after_graph_replays(sp, torch):  # noqa: F811
    """A replayed graph writes LDCAs unseen by the host: the reset of a router
    that looks untouched still zeroes all of it."""
    kw = dict(BASE, k_log2=8, lr=3, lc_log2=6, n_routers=2)
    x = _pairs("planes", 3)
    t = dev(torch, x)
    rec = np.zeros(1, sp.BATCH)
    rec[0] = (t.data_ptr(), x.shape[0], 0, 0)
    tab = torch.from_numpy(rec.view(np.uint8)).cuda()
    with sp.SuperPoint(**kw) as ctx:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
            sp.sp_update_batched_device(ctx.ctx, tab, 1)
        sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
        for _ in range(2):
            sp.sp_reset_range(ctx.ctx, 0, 2)
            g.replay()
            assert_same_sketch(ctx, O.Sketch(oracle_params(kw)).update(x), 0)
            sp.sp_reset(ctx.ctx, 0)
            seav, ldca = ctx.sketch_image(0)
            assert not seav.any() and not ldca.any()


def test_recorded_merge_then_calls_on_its_sources(sp, torch):  # noqa: F811
    """A graph of a binned update and a merge, replayed between resets: the
    source's bits are found by calls after the replay, not only the merged ones."""
    kw = dict(BASE, k_log2=8, lr=3, lc_log2=6, n_routers=3, scan_mode=2)
    op = oracle_params(kw)
    x, y = _pairs("planes", 4), _pairs("planes", 5)
    t, u = dev(torch, x), dev(torch, y)
    with sp.SuperPoint(**kw) as ctx:
        sp.sp_reserve(ctx.ctx)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
            ctx.update(t, router=0)
            ctx.merge([0, 2], 1)
        sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
        for _ in range(2):
            sp.sp_reset_range(ctx.ctx, 0, 3)
            ctx.update(u, router=2)                       # pending when the replay merges
            g.replay()
            assert_same_sketch(ctx, O.Sketch(op).update(x), 0)
            assert_same_sketch(ctx, O.Sketch(op).update(y), 2)
            ctx.merge([0, 2], 1)
            assert_same_sketch(ctx, O.Sketch(op).update(x).update(y), 1)
