"""eco_write_params / eco_read_params where their tiles and chunks can go
wrong: packed, padded and very long rows, one slot, a run of slots longer than
one staging chunk, and the values at the ends of the range.  What was written
comes back bit for bit, slots beside the run keep theirs, and the streamed
copy equals the oracle's quantiser."""
import numpy as np
import pytest

import oracle
from paper_2510_18221_gb300 import workloads
from tests import harness, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("key,slots,slot0,n,kw", [
    ("small", 9, 0, 9, dict(patch_k=0, hidden=128)),
    ("mid", 40, 3, 1, dict(patch_k=1, hidden=32)),
    ("paperform", 33, 1, 31, dict(n_hidden=4)),
    ("ecology", 5, 2, 3, dict(patch_k=31, view="front")),
    ("terrain", 4, 0, 3, dict(patch_k=31, hidden=32)),
    ("mid", 700, 50, 640, dict()),                                   # three staging chunks
])
def test_params_round_trip(key, slots, slot0, n, kw, prec):
    from paper_2510_18221_gb300 import eco
    w = workloads.scaled(key, 64, slots, 0, precision=prec, **kw)
    env, orc = eco.Env(w), oracle.Oracle(w)
    env.reset()
    rows = inputs.random_params(env.P, n, seed=slots)
    rows[0, ::7] = 0.0
    rows[-1, ::5] = np.float32(-3.0e38)
    rows[-1, 1::5] = np.float32(1.0e-42)
    env.write_params(0, slot0, rows)
    got = env.read_params(0)
    assert np.array_equal(got[slot0:slot0 + n].view(np.uint32), rows.view(np.uint32))
    assert not got[:slot0].any() and not got[slot0 + n:].any()
    assert np.array_equal(env.read_params(0, slot0, n).view(np.uint32), rows.view(np.uint32))
    keep = range(slot0, slot0 + n) if n < 100 else (slot0, slot0 + n // 2, slot0 + n - 1)
    harness.check_streamed(env, orc, {s: rows[s - slot0] for s in keep})
    env.close()
