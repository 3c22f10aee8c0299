"""The batched direct scan's chunk tickets, against the oracle: no chunk, fewer
chunks than blocks, one more than the blocks, many per block, batches that the
kernel skips, launches in a row (the counter is zero again after each), every
block size, and replays of a captured launch over a rewritten table.
"""
import numpy as np
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_sketch, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

KW = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), k_log2=8, lr=3, lc_log2=9, theta=64, seed=111, scan_mode=1, n_routers=3)
BLOCKS = 152 * 8                      # resident 256-thread blocks on a GB300; chunks of 2,048 pairs


def _table(sp, torch, entries):  # noqa: F811
    rec = np.zeros(max(1, len(entries)), sp.BATCH)
    for i, e in enumerate(entries):
        rec[i] = (*e, 0)
    return torch.from_numpy(rec.view(np.uint8)).cuda()


@pytest.mark.parametrize("sizes", [[0, 0], [1], [2048, 2049], [BLOCKS * 2048], [BLOCKS * 2048 + 1],
                                   [100000] * 40, [3, 0, 2 * BLOCKS * 2048 + 5, 7]])
def test_launches_in_a_row(sp, torch, sizes):  # noqa: F811
    rng = np.random.default_rng(len(sizes))
    parts = [W.uniform_pairs(n, seed=1100 + i, n_hosts=max(1, n // 20)) for i, n in enumerate(sizes)]
    tens = [dev(torch, p, 0) if len(p) else torch.zeros(4, dtype=torch.int32, device="cuda") for p in parts]
    with sp.SuperPoint(**KW) as ctx:
        osks = [O.Sketch(oracle_params(KW)) for _ in range(3)]
        for _ in range(3):
            routers = rng.integers(0, 3, len(sizes)).tolist()
            entries = [(t.data_ptr(), len(p), r) for t, p, r in zip(tens, parts, routers)]
            table = _table(sp, torch, entries)
            sp.sp_update_batched_device(ctx.ctx, table, len(entries))
            for p, r in zip(parts, routers):
                osks[r].update(p)
        for r in range(3):
            assert_same_sketch(ctx, osks[r], r)


def test_after_a_table_of_skipped_batches(sp, torch):  # noqa: F811
    x = W.uniform_pairs(50000, seed=3, n_hosts=900)
    t = dev(torch, x)
    with sp.SuperPoint(**KW) as ctx:
        bad = _table(sp, torch, [(t.data_ptr(), len(x), 9), (t.data_ptr(), len(x), 7)])
        good = _table(sp, torch, [(t.data_ptr(), len(x), 9), (t.data_ptr(), len(x), 1)])
        for table in (bad, good, bad):
            sp.sp_update_batched_device(ctx.ctx, table, 2)
        assert_same_sketch(ctx, O.Sketch(oracle_params(KW)).update(x), 1)
        sp.sp_autotune(ctx.ctx, t)                              # every block size and grid
        sp.sp_update_batched(ctx.ctx, [2], [t])
        assert_same_sketch(ctx, O.Sketch(oracle_params(KW)).update(x), 2)


def test_replays_over_a_rewritten_table(sp, torch):  # noqa: F811
    pool = [W.uniform_pairs(n, seed=1200 + n, n_hosts=400) for n in (10, 300000, 4096)]
    tens = [dev(torch, p) for p in pool]
    table = _table(sp, torch, [(tens[0].data_ptr(), len(pool[0]), 0)])
    with sp.SuperPoint(**KW) as ctx:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
            sp.sp_update_batched_device(ctx.ctx, table, 1)
        sp.sp_set_stream(ctx.ctx, torch.cuda.current_stream())
        osk = O.Sketch(oracle_params(KW))
        for p, t in zip(pool, tens):
            table.copy_(_table(sp, torch, [(t.data_ptr(), len(p), 0)]))
            g.replay()
            assert_same_sketch(ctx, osk.update(p), 0)
