"""Detects of SEAs with more tuples than the queue of hosts to be tested holds,
against the oracle: hosts tested turn by turn, and in one lane when a single
turn fills the queue, for LDC lines of one word, two, four and more.
"""
import pytest

import oracle as O
from test_detect_forms_gpu import PROFILES, _pairs
from test_parity_gpu import assert_same_results, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu


# hosts in one SEA: a few turns of the join, and turns of more than 256 tuples each
@pytest.mark.parametrize("hosts", [9, 17, 40])
@pytest.mark.parametrize("k_log2", [5, 6, 7, 12])
@pytest.mark.parametrize("p", [0, 3, 4, 5])                    # four rows of 128, three rows, two rows staged and not
def test_queue_of_one_sea(sp, torch, p, k_log2, hosts):  # noqa: F811
    kw = dict(PROFILES[p], k_log2=k_log2, lr=2, lc_log2=9, theta=16, seed=131 + p)
    x = _pairs(kw, hosts, 60, 1, 1310 + hosts)
    with sp.SuperPoint(**kw) as ctx, sp.SuperPoint(**dict(kw, window_slices=2)) as slid:
        ctx.update(dev(torch, x))
        slid.update(dev(torch, x[::2].copy()))
        slid.slide()
        slid.update(dev(torch, x[1::2].copy()))
        want, n_want, _ = O.Sketch(oracle_params(kw)).update(x).detect()
        for c in (ctx, slid):
            got, n, rc = c.detect()
            assert rc == sp.SP_OK and n == n_want
            assert_same_results(got, want)
