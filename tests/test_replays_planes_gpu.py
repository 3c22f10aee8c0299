"""Replays of recorded binned updates in contexts whose plane accumulators
already held bits when the capture began, against the oracle.

A program warms up before it captures, and a merge leaves its sources' planes
pending.  What a recorded call finds in the planes is decided when it runs:
after a reset, an import or a closed slice the bits of earlier windows are gone,
whatever the host knew at the capture.
"""
import numpy as np
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_results, assert_same_sketch, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

N = 2003
SHAPE = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), lr=3, lc_log2=6, theta=64, scan_mode=2)


def _pairs(i):
    return W.uniform_pairs(N, seed=900 + i, n_hosts=24)


class Recorded:
    """A graph of `calls(ctx)`, captured on a side stream; the context goes back to the current one."""

    def __init__(self, sp, torch, ctx, calls):  # noqa: F811
        torch.cuda.synchronize()
        self.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(self.graph):
            sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
            calls(ctx)
        sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())

    def replay(self):
        self.graph.replay()


@pytest.mark.parametrize("k_log2", [6, 8])
@pytest.mark.parametrize("form", ["update", "update+detect", "update+merge+detect", "reset+update+merge+detect"])
def test_windows_after_an_eager_merge(sp, torch, form, k_log2):  # noqa: F811
    kw = dict(SHAPE, k_log2=k_log2, seed=91, n_routers=2)
    op = oracle_params(kw)
    buf = dev(torch, _pairs(0))

    def calls(ctx):
        if "reset" in form:
            sp.sp_reset_range(ctx.ctx, 0, 2)
        ctx.update(buf, router=0)
        if "merge" in form:
            ctx.merge([0], 1)
        if "detect" in form:
            sp.sp_detect_async(ctx.ctx, 1 if "merge" in form else 0, 64)

    with sp.SuperPoint(**kw) as ctx:
        ctx.update(dev(torch, _pairs(1)), router=0)                 # the warm-up
        ctx.merge([0], 1)
        ctx.detect(1, 64)
        g = Recorded(sp, torch, ctx, calls)
        for w in (2, 3, 4):
            x = _pairs(w)
            osk = O.Sketch(op).update(x)
            buf.copy_(dev(torch, x))
            if "reset" not in form:
                sp.sp_reset_range(ctx.ctx, 0, 2)
            g.replay()
            if "detect" in form:
                got, n, _ = sp.sp_results(ctx.ctx)
                want, n_want, _ = osk.detect(64)
                assert n == n_want
                assert_same_results(got, want)
            assert_same_sketch(ctx, osk, 0)
            assert_same_sketch(ctx, osk if "merge" in form else O.Sketch(op), 1)
        y = _pairs(9)                                               # no reset: the window goes on
        buf.copy_(dev(torch, y))
        if "reset" not in form:
            g.replay()
            assert_same_sketch(ctx, osk.update(y), 0)
            ctx.merge([0], 1)
            assert_same_sketch(ctx, osk, 1)


def test_recorded_fold_of_a_window_long_gone(sp, torch):  # noqa: F811
    """Only the detect is recorded, while the warm-up's planes are pending."""
    kw = dict(SHAPE, k_log2=8, seed=92, n_routers=2)
    with sp.SuperPoint(**kw) as ctx:
        ctx.update(dev(torch, _pairs(1)), router=0)
        ctx.merge([0], 1)
        g = Recorded(sp, torch, ctx, lambda c: sp.sp_detect_async(c.ctx, 0, 64))
        for w in (2, 3):
            sp.sp_reset_range(ctx.ctx, 0, 2)
            g.replay()
            assert sp.sp_results(ctx.ctx)[1] == 0
            assert_same_sketch(ctx, O.Sketch(oracle_params(kw)), 0)
            x = _pairs(w)
            ctx.update(dev(torch, x), router=0)
            g.replay()
            osk = O.Sketch(oracle_params(kw)).update(x)
            assert_same_results(sp.sp_results(ctx.ctx)[0], osk.detect(64)[0])
            assert_same_sketch(ctx, osk, 0)


def test_replay_after_an_import(sp, torch):  # noqa: F811
    kw = dict(SHAPE, k_log2=8, seed=93, n_routers=2)
    op = oracle_params(kw)
    x, y = _pairs(5), _pairs(6)
    buf = dev(torch, x)
    with sp.SuperPoint(**kw) as other:
        other.update(dev(torch, y))
        image = sp.sp_export(other.ctx, 0)
    with sp.SuperPoint(**kw) as ctx:
        ctx.update(dev(torch, _pairs(1)), router=0)
        ctx.merge([0], 1)
        g = Recorded(sp, torch, ctx, lambda c: c.update(buf, router=0))
        for _ in range(2):
            assert sp.sp_import(ctx.ctx, 0, image) == sp.SP_OK
            g.replay()
            assert_same_sketch(ctx, O.Sketch(op).update(x).update(y), 0)


def test_recorded_slices_after_pending_planes(sp, torch):  # noqa: F811
    """Sliding: the slice that was open at the capture is over after the first
    replayed slide, its bits with it once the window has passed."""
    kw = dict(SHAPE, k_log2=8, seed=94, window_slices=2)
    op = oracle_params(kw)
    buf = dev(torch, _pairs(0))
    with sp.SuperPoint(**kw) as ctx:
        slices = [[1]]
        ctx.update(dev(torch, _pairs(1)))                           # pending when the capture begins

        def calls(c):
            c.update(buf)
            c.slide()

        g = Recorded(sp, torch, ctx, calls)
        for w in (2, 3, 4, 5):
            buf.copy_(dev(torch, _pairs(w)))
            g.replay()
            slices[-1].append(w)
            slices.append([])
            osk = O.Sketch(op)
            for i in slices[-2] + slices[-1]:
                osk.update(_pairs(i))
            got, n, _ = ctx.detect(0, 64)
            want, n_want, _ = osk.detect(64)
            assert n == n_want
            assert_same_results(got, want)
            assert_same_sketch(ctx, osk)
