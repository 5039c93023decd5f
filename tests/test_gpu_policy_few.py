"""The register form of the policy kernel with few agents (its weights
requested into L1 ahead, agents spread over the CTAs) against the ring form
(variant 3), bit for bit: logits, actions, state and statistics, on both sides
of three eighths of the launch's warps, with blocks shorter than what is
requested ahead, and with the last agents in the workspace's last slots."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads
from tests import harness

pytestmark = pytest.mark.gpu

SHAPES = [
    ("small", dict(patch_k=0, n_scalars=4, precision="fp8")),     # blocks of a few hundred bytes
    ("mid", dict(precision="fp32")),
    ("mid", dict(precision="bf16", patch_k=9)),
    ("mid", dict(precision="fp8", patch_k=15, hidden=128)),
    ("terrain", dict(precision="bf16")),
]


@pytest.mark.parametrize("variant", [1, 2, 4, 5, 6, 9, 10])
@pytest.mark.parametrize("key,kw", SHAPES)
def test_few_equals_ring(key, kw, variant):
    import torch
    from paper_2510_18221_gb300 import eco
    warps = {1: 40, 2: 40, 4: 32, 5: 32, 6: 32, 9: 36, 10: 36}[variant]    # resident per SM at most
    edge = 3 * warps * torch.cuda.get_device_properties(0).multi_processor_count // 8
    for n in (1, 33, edge, edge + 1):
        w = workloads.scaled(key, 160, n, n, **kw)
        a, b = eco.Env(w, policy_variant=variant), eco.Env(w, policy_variant=3)
        for x in (a, b):
            x.reset()
            x.step(2)
        la, aa = a.read_policy_io(0)
        lb, ab = b.read_policy_io(0)
        assert np.array_equal(la.view(np.uint32), lb.view(np.uint32)) and np.array_equal(aa, ab), n
        sa, sb = a.read_state(0), b.read_state(0)
        for k in harness.STATE_KEYS:
            assert np.array_equal(sa[k], sb[k]), (k, n)
        assert a.stats() == b.stats()
        a.close()
        b.close()
