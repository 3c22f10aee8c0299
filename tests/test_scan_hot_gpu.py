"""The direct scan with heavy hosts held on chip, against the oracle: windows
with one host for nearly all pairs, more heavy hosts than vectors, hosts that
share a table slot, the address that marks a free slot, repeated pairs, every
estimator width, and sizes around the line from which the form is used.
"""
import numpy as np
import pytest

import oracle as O
from paper_1901_07306_gb300 import workloads as W
from test_parity_gpu import assert_same_sketch, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

LINE = 1 << 18
KW = dict(r=12, isb=(0, 7, 14), ibn=(8, 8, 8), theta=64, seed=91, scan_mode=1)


def _heavy(n, hosts, share, seed, peers=2**32):
    """n pairs, a share of them from the given hosts (evenly), the rest uniform."""
    rng = np.random.default_rng(seed)
    x = W.uniform_pairs(n, seed=seed)
    at = rng.random(n) < share
    x[at, 0] = np.asarray(hosts, np.uint32)[rng.integers(0, len(hosts), int(at.sum()))]
    x[at, 1] = rng.integers(0, peers, int(at.sum()), dtype=np.uint64).astype(np.uint32)
    return x


@pytest.mark.parametrize("k_log2,lr,lc_log2", [(5, 1, 0), (6, 3, 7), (10, 4, 12), (12, 8, 8), (16, 2, 4)])
@pytest.mark.parametrize("n,off", [(LINE - 1, 0), (LINE, 1), (LINE + 1, 0), (700003, 1)])
def test_sizes_and_widths(sp, torch, k_log2, lr, lc_log2, n, off):  # noqa: F811
    kw = dict(KW, k_log2=k_log2, lr=lr, lc_log2=lc_log2)
    hosts = [0xFFFFFFFF, 0, 5] + list(range(1000, 1100))
    x = _heavy(n, hosts, 0.7, k_log2 * 10 + off)
    with sp.SuperPoint(**kw) as ctx:
        ctx.update(dev(torch, x, off))
        assert_same_sketch(ctx, O.Sketch(oracle_params(kw)).update(x))


@pytest.mark.parametrize("hosts,share,peers", [([7], 1.0, 2**32), ([0xFFFFFFFF], 1.0, 2**32), ([7], 1.0, 1),
                                               (list(range(64)), 1.0, 2**32), (list(range(65, 2400)), 1.0, 50),
                                               ([3, 9, 11], 0.02, 2**32)])
def test_heavy_hosts(sp, torch, hosts, share, peers):  # noqa: F811
    kw = dict(KW, k_log2=10, lr=4, lc_log2=10)
    x = _heavy(500001, hosts, share, len(hosts), peers)
    with sp.SuperPoint(**kw) as ctx:
        ctx.update(dev(torch, x))
        osk = O.Sketch(oracle_params(kw)).update(x)
        assert_same_sketch(ctx, osk)
        got, n, _ = ctx.detect()
        want, n_want, _ = osk.detect()
        assert n == n_want and np.array_equal(got, want)


def test_slots_shared_by_hosts(sp, torch):  # noqa: F811
    """Heavy hosts whose table slots collide (slot = top 11 bits of the host
    times an odd constant): only one of them can be held."""
    inv = pow(0x9E3779B1, -1, 1 << 32)
    hosts = [((5 << 21) + j) * inv % (1 << 32) for j in range(1, 9)]
    assert len({(h * 0x9E3779B1 % (1 << 32)) >> 21 for h in hosts}) == 1
    kw = dict(KW, k_log2=8, lr=3, lc_log2=8)
    x = _heavy(400000, hosts, 0.9, 17)
    with sp.SuperPoint(**kw) as ctx:
        ctx.update(dev(torch, x))
        assert_same_sketch(ctx, O.Sketch(oracle_params(kw)).update(x))
