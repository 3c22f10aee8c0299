"""Batched direct scans of one context that may run at the same time, against
the oracle: calls on two streams without a wait between them, and replays of a
recorded table scan beside an eager one.  Setting a bit is idempotent and order
independent, so neither may lose a pair, nor may the next launch.
"""
import numpy as np
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_sketch, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

KW = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), k_log2=8, lr=3, lc_log2=9, theta=64, seed=121, scan_mode=1, n_routers=3)
# about 2,900 chunks of 2,048 pairs over the host link: both launches have chunks left while the other one draws
SIZES = [(150001, 151000), (149001, 152000), (40000, 41003)]
PARTS = 20


@pytest.fixture(scope="module")
def streams(torch):  # noqa: F811
    out = []
    for r, (lo, hi) in enumerate(SIZES):
        rng = np.random.default_rng(1300 + r)
        parts = [W.uniform_pairs(int(n), seed=1400 + 100 * r + i, n_hosts=5000)
                 for i, n in enumerate(rng.integers(lo, hi, PARTS))]
        osk = O.Sketch(oracle_params(KW))
        for p in parts:
            osk.update(p)
        tens = [torch.from_numpy(p.reshape(-1).view(np.int32)).pin_memory() for p in parts]
        rec = np.zeros(PARTS, sp_batch())
        for i, t in enumerate(tens):
            rec[i] = (t.data_ptr(), t.numel() // 2, r, 0)
        out.append((tens, torch.from_numpy(rec.view(np.uint8)).cuda(), osk))
    return out


def sp_batch():
    from paper_1901_07306_gb300 import sp as mod
    return mod.BATCH


def _send(sp, ctx, streams, r, form):  # noqa: F811
    if form == "table":
        sp.sp_update_batched_device(ctx.ctx, streams[r][1], PARTS)
    else:
        sp.sp_update_batched(ctx.ctx, [r] * PARTS, streams[r][0])


@pytest.mark.parametrize("form", ["table", "batched"])
def test_two_streams(sp, torch, streams, form):  # noqa: F811
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with sp.SuperPoint(**KW) as ctx:
        for _ in range(4):
            sp.sp_reset_range(ctx.ctx, 0, 3)
            torch.cuda.synchronize()
            for r, s in ((0, a), (1, b)):
                sp.sp_set_stream(ctx.ctx, s)
                _send(sp, ctx, streams, r, form)
            torch.cuda.synchronize()
            _send(sp, ctx, streams, 2, form)
            torch.cuda.synchronize()
            for r in range(3):
                assert_same_sketch(ctx, streams[r][2], r)


@pytest.mark.parametrize("form", ["table", "batched"])
def test_replay_beside_an_eager_call(sp, torch, streams, form):  # noqa: F811
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with sp.SuperPoint(**KW) as ctx:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
            _send(sp, ctx, streams, 0, "table")
        sp.sp_set_stream(ctx.ctx, b)
        for _ in range(4):
            sp.sp_reset_range(ctx.ctx, 0, 3)
            torch.cuda.synchronize()
            with torch.cuda.stream(a):
                g.replay()
            _send(sp, ctx, streams, 1, form)
            torch.cuda.synchronize()
            _send(sp, ctx, streams, 2, form)
            torch.cuda.synchronize()
            for r in range(3):
                assert_same_sketch(ctx, streams[r][2], r)
