"""Contexts of different sizes, one per host thread, whose calls launch the
same kernels with different amounts of shared memory at the same time.
"""
import threading

import numpy as np
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_sketch, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

N = 20011
BASE = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), lr=4, theta=64)
# the plane pass of a fixed LC: its list counts follow k and the staging shape
PLANES = [dict(BASE, k_log2=k, lc_log2=14, seed=141 + k, scan_mode=2) for k in (10, 5, 8, 5)]
# the plane pass of any LC: its rows follow LC too
ANY_LC = [dict(BASE, k_log2=k, lc_log2=lc, seed=151 + k, scan_mode=2) for k, lc in ((10, 5), (6, 12), (5, 13), (8, 7))]


def _in_threads(work, count):
    errors = []

    def body(i):
        try:
            work(i)
        except Exception as e:  # noqa: BLE001  handed to the test's thread
            errors.append(e)

    threads = [threading.Thread(target=body, args=(i,)) for i in range(count)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("forms", [PLANES, ANY_LC], ids=["fixed_lc", "any_lc"])
def test_plane_passes_of_several_sizes(sp, torch, forms):  # noqa: F811
    pairs = [W.uniform_pairs(N, seed=1500 + i, n_hosts=900) for i in range(len(forms))]
    tens = [dev(torch, p) for p in pairs]
    ctxs = [sp.SuperPoint(**kw) for kw in forms]
    for i, c in enumerate(ctxs):
        sp.sp_reserve(c.ctx)
        sp.sp_set_binned_shape(c.ctx, [0, 2, 0, 0][i])
    torch.cuda.synchronize()

    def work(i):
        for _ in range(3000):
            ctxs[i].update(tens[i])

    _in_threads(work, len(forms))
    torch.cuda.synchronize()
    for c, kw, p in zip(ctxs, forms, pairs):
        assert_same_sketch(c, O.Sketch(oracle_params(kw)).update(p))
        c.close()


def test_tables_of_several_lengths(sp, torch):  # noqa: F811
    counts = [1, 8192, 700, 5000]                # batches of a call: the table's prefix is in shared memory
    kw = dict(BASE, k_log2=8, lc_log2=9, seed=161, scan_mode=1)
    pairs = [W.uniform_pairs(n, seed=1600 + n, n_hosts=500) for n in counts]
    tens = [dev(torch, p) for p in pairs]
    tables = []
    for n, t in zip(counts, tens):
        rec = np.zeros(n, sp.BATCH)              # one pair a batch
        rec["pairs"] = t.data_ptr() + 8 * np.arange(n, dtype=np.uint64)
        rec["n_pairs"] = 1
        tables.append(torch.from_numpy(rec.view(np.uint8)).cuda())
    ctxs = [sp.SuperPoint(**kw) for _ in counts]
    torch.cuda.synchronize()

    def work(i):
        for _ in range(2000):
            sp.sp_update_batched_device(ctxs[i].ctx, tables[i], counts[i])

    _in_threads(work, len(counts))
    torch.cuda.synchronize()
    for c, p in zip(ctxs, pairs):
        assert_same_sketch(c, O.Sketch(oracle_params(kw)).update(p))
        c.close()
