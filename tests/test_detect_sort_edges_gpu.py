"""The result sort of the detect at the edges of its forms.

k_sort_emit sorts up to 2,048 keys in one block, more as runs of 2,048 merged
16 at a time (one round up to 32,768 keys, two above).  A result buffer of
exactly the edge sizes makes the sort run with that many keys: the list is then
an unspecified subset of the oracle's, in ascending order, each record bit for
bit.
"""
import numpy as np
import pytest

import oracle as O
from test_parity_gpu import _many_hosts, dev, oracle_params, sp, torch  # noqa: F401

pytestmark = pytest.mark.gpu

KW = dict(r=16, isb=(0, 8), ibn=(9, 9), theta=32, seed=57)
_WANT = {}


def _want():
    if not _WANT:
        pairs, _ = _many_hosts(40000, 57)
        want, n, overflow = O.Sketch(oracle_params(KW)).update(pairs).detect()
        assert not overflow and n > 36000
        _WANT.update(pairs=pairs, want=want, n=n)
    return _WANT


@pytest.mark.parametrize("cap", [1, 2, 31, 33, 2047, 2048, 2049, 4096, 32767, 32768, 32769, 36000])
def test_sort_edges(sp, torch, cap):  # noqa: F811
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
