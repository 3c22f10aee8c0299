"""The detect's forms -- SEAs of four rows of 128 SEs (one lane per 16 SEs),
other staged SEAs, SEAs read from global memory -- against the oracle, around
the lines between them (1 KiB, a size that 16 does not divide), with
SEAs from empty to crowded, in discrete and sliding windows.
"""
import numpy as np
import pytest

import oracle as O
from test_parity_gpu import assert_same_results, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

FOUR = (7, 7, 7, 7)
PROFILES = [dict(r=8, isb=(0, 6, 12, 18), ibn=FOUR),           # 24 LP bits, the most four such rows cover
            dict(r=14, isb=(0, 5, 10, 15), ibn=FOUR),
            dict(r=16, isb=(0, 4, 8, 12), ibn=FOUR),
            dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8)),         # 768 bytes
            dict(r=16, isb=(0, 8), ibn=(9, 9)),                # 1,024 bytes
            dict(r=14, isb=(0, 9), ibn=(10, 10)),              # 2,048 bytes: global memory
            dict(r=24, isb=(0, 4), ibn=(5, 5)),                # 64 bytes
            dict(r=24, isb=(0, 3, 6), ibn=(4, 4, 3))]          # 40 bytes: global memory


def _pairs(kw, hosts, peers, crowd, seed):
    """hosts x peers distinct-ish pairs; crowd > 0: the hosts share that many SEAs."""
    rng = np.random.default_rng(seed)
    h = rng.integers(0, 2**32, hosts, dtype=np.uint32)
    if crowd:
        h = (h & ~np.uint32((1 << kw["r"]) - 1)) | rng.integers(0, crowd, hosts, dtype=np.uint32)
    hip = np.repeat(h, peers)
    x = np.stack([hip, rng.integers(0, 2**32, hip.size, dtype=np.uint32)], 1)
    return np.ascontiguousarray(x[rng.permutation(hip.size)])


# 2^24 SEAs take the oracle seconds: one traffic each
CASES = [(p, h, c) for p, prof in enumerate(PROFILES) for h, c in [(700, 0), (1, 0), (60, 5), (40, 1)]
         if prof["r"] < 24 or (h, c) == (700, 0)]


@pytest.mark.parametrize("p,hosts,crowd", CASES)
def test_forms(sp, torch, p, hosts, crowd):  # noqa: F811
    kw = dict(PROFILES[p], k_log2=8, lr=3, lc_log2=12, theta=16, seed=101 + p)
    x = _pairs(kw, hosts, 40, crowd, 1010 + p)
    with sp.SuperPoint(**kw) as ctx, sp.SuperPoint(**dict(kw, window_slices=3)) as slid:
        ctx.update(dev(torch, x))
        slid.update(dev(torch, x[::2].copy()))
        slid.slide()
        slid.update(dev(torch, x[1::2].copy()))
        want, n_want, _ = O.Sketch(oracle_params(kw)).update(x).detect()
        assert n_want >= min(hosts, 1)
        for c in (ctx, slid):
            got, n, rc = c.detect()
            assert rc == sp.SP_OK and n == n_want
            assert_same_results(got, want)
