"""The result sort at the lines of its merge rounds, against the oracle.

k_sort_emit sorts runs of 2,048 keys and merges up to 8 of them a round: two,
four and eight runs take different code, 8 runs one round, 64 two, more three,
and an odd number of rounds starts in the other buffer.  A result buffer of
exactly the edge sizes makes the sort run with that many keys: the list is then
an unspecified subset of the oracle's, in ascending order, each record bit for
bit.
"""
import numpy as np
import pytest

import oracle as O
from test_parity_gpu import _many_hosts, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

KW = dict(r=16, isb=(0, 8), ibn=(9, 9), theta=32, seed=58)
_WANT = {}


def _want():
    if not _WANT:
        pairs, _ = _many_hosts(150000, 58)
        want, n, overflow = O.Sketch(oracle_params(KW)).update(pairs).detect()
        assert not overflow and n > 132000
        _WANT.update(pairs=pairs, want=want, n=n)
    return _WANT


@pytest.mark.parametrize("cap", [4095, 4096, 4097, 8191, 8192, 8193, 16383, 16384, 16385, 20481, 131071, 131072, 131073])
def test_merge_rounds(sp, torch, cap):  # noqa: F811
    w = _want()
    with sp.SuperPoint(max_candidates=cap, **KW) as ctx:
        ctx.update(dev(torch, w["pairs"]))
        got, n, rc = ctx.detect()
    assert rc == sp.SP_ERR_CANDIDATE_OVERFLOW and n == w["n"] and len(got) == cap
    assert np.all(got["ip"][1:] > got["ip"][:-1])
    at = np.searchsorted(w["want"]["ip"], got["ip"])
    for f in ("ip", "z0", "flags"):
        assert np.array_equal(got[f], w["want"][f][at]), f
    assert np.array_equal(got["est"].view(np.uint64), w["want"]["est"][at].view(np.uint64))
