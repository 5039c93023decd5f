"""The ring form of the policy kernel (variants 3 and 7) against the register
form of the same family (6 and 8), bit for bit: logits, actions, state and
statistics.  Populations below, at and above one round of the launch's warps;
blocks with fewer batches than the ring (which fall back to the register
form), with one batch more, and with several hidden layers; patches inside the
world and across its seams, larger than the short cut of the sparse list, and
the rules whose observation it does not cover."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads
from tests import harness

pytestmark = pytest.mark.gpu

SHAPES = [
    ("small", dict(patch_k=3, precision="fp8")),                       # fewer batches than the ring
    ("small", dict(patch_k=5, hidden=64, precision="fp8", n_scalars=4)),
    ("mid", dict(precision="fp32")),
    ("mid", dict(precision="bf16", flags=())),                         # an unrotated patch
    ("mid", dict(precision="fp8", patch_k=13)),                        # 169 cells: past the sparse list's 128
    ("mid", dict(precision="fp8", view="front", wall_density=0.3)),
    ("mid", dict(precision="bf16", patch_k=0, hidden=128)),            # no vision
    ("paperform", dict(precision="fp8", n_hidden=3, hidden=128)),
    ("ecology", dict(precision="bf16", view="front")),
    ("terrain", dict(precision="fp32", hidden=32)),
]


@pytest.mark.parametrize("pair", [(6, 3), (8, 7)])
@pytest.mark.parametrize("key,kw", SHAPES)
def test_ring_equals_register_form(key, kw, pair):
    from paper_2510_18221_gb300 import eco
    for side, n in ((32, 1), (32, 37), (30, 300), (160, 3100)):
        if side * side < 8 * n and key == "terrain":
            continue
        w = workloads.scaled(key, side, n + n // 4, n, **kw)
        a, b = (eco.Env(w, policy_variant=v) for v in pair)
        for x in (a, b):
            x.reset()
            x.step(3)
        la, aa = a.read_policy_io(0)
        lb, ab = b.read_policy_io(0)
        assert np.array_equal(la.view(np.uint32), lb.view(np.uint32)) and np.array_equal(aa, ab), (side, n)
        sa, sb = a.read_state(0), b.read_state(0)
        for k in harness.STATE_KEYS:
            assert np.array_equal(sa[k], sb[k]), (k, side, n)
        assert a.stats() == b.stats()
        a.close()
        b.close()
