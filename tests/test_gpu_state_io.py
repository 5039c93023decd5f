"""eco_read_state through its three routes -- packed into pinned memory, arrays
copied one by one, and pieces of the staging region -- for sides and slot
counts that leave ragged ends, worlds at odd offsets inside a batch, and views
that ask for some arrays only.  Every array equals the oracle's after reset."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2510_18221_gb300 import workloads
from tests import harness

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("key,sizes", [
    ("small", [(4, 3, 2)]),
    ("mid", [(62, 701, 333), (6, 1, 1), (64, 257, 200)]),
    ("terrain", [(50, 333, 300)]),
    ("ecology", [(212, 2001, 1500), (256, 4097, 4000)]),       # around one megabyte
    ("small", [(1024, 5, 5)]),                                  # a staging region smaller than the cells
])
def test_read_state_equals_the_oracle(key, sizes):
    from paper_2510_18221_gb300 import eco
    ws = [workloads.scaled(key, side, slots, alive, seed=i, patch_k=3, hidden=32)
          for i, (side, slots, alive) in enumerate(sizes)]
    env = eco.Env(ws)
    env.reset()
    for e, w in enumerate(ws):
        orc = oracle.Oracle(w)
        orc.reset()
        got = env.read_state(e)
        harness.compare_state(got, orc, "world %d" % e)
        assert np.array_equal(got["colour"], orc.colour)
        # some arrays only: the others are left alone
        part = {"occ": np.full(w["side"] ** 2, -7, np.int32), "y": np.full(w["slots"], -7, np.int32),
                "alive": np.full(w["slots"], 9, np.uint8)}
        v = eco.eco_state_view(**{k: a.ctypes.data for k, a in part.items()})
        assert eco.lib().eco_read_state(env.h, e, ctypes.byref(v)) == eco.ECO_OK
        for k, a in part.items():
            assert np.array_equal(a, got[k]), k
    env.close()
