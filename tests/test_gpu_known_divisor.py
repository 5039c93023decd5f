"""The founders' weights of the plain form on the device, bit for bit: each is
the IEEE quotient of its normal by sqrt(fan-in) (csrc/eco_params.cu,
divide_by_known; the head's by an IEEE division).

The normal of logical parameter p of a slot depends on the seed, the slot and p
alone, so one shape gives it for all the others: 4-64-64-A, whose divisors 2
and 8 are powers of two and leave the normal's digits as they are."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads

pytestmark = pytest.mark.gpu

SLOTS = 500


def _founders(key, prec, **kw):
    from paper_2510_18221_gb300 import eco
    env = eco.Env(workloads.scaled(key, 64, SLOTS, SLOTS, seed=3, precision=prec, wall_density=0.0,
                                   policy_form="plain", **kw))
    env.reset()
    w, D, H, A = env.read_params(0), env.D, env.H, env.A
    env.close()
    # (first parameter, count, fan-in) of the weight sections
    return w, [(0, H * D, D), (H * D + H, H * H, H), (H * D + 2 * H + H * H, A * H, H)]


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
def test_founders_weights_are_ieee_quotients(prec):
    raw, sections = _founders("mid", prec, patch_k=0, n_scalars=4, hidden=64)
    normal = np.full(raw.shape[1], np.nan, np.float32)[None].repeat(SLOTS, 0)
    for p, n, fan in sections:
        normal[:, p:p + n] = raw[:, p:p + n] * np.float32(np.sqrt(fan))      # exact: 2 or 8
    seen = set()
    for key, kw in [("mid", dict(patch_k=k, n_scalars=s, hidden=h)) for k, s, h in (
            (0, 8, 32), (1, 4, 32), (1, 8, 64), (3, 4, 128), (5, 8, 32), (7, 4, 64), (11, 8, 64), (13, 8, 32), (15, 8, 128),
            (31, 4, 32))] + [("terrain", dict(patch_k=5, hidden=64)), ("terrain", dict(patch_k=1, hidden=128))]:
        w, sections = _founders(key, prec, **kw)
        for p, n, fan in sections:
            n = min(n, normal.shape[1] - p)
            if n <= 0:
                continue
            z = normal[:, p:p + n]
            known = ~np.isnan(z)
            want = z / np.sqrt(np.float32(fan))
            assert want.dtype == np.float32
            got = w[:, p:p + n]
            assert np.array_equal(got[known].view(np.uint32), want[known].view(np.uint32)), (key, kw, p, fan)
            if known.any():
                seen.add(fan)
    # every kind of fan-in: D of 3 k^2 + 4, 3 k^2 + 8, 4 k^2 + 16, and each H
    assert {7, 8, 11, 31, 83, 151, 371, 515, 683, 2887, 116, 20, 32, 64, 128} <= seen
