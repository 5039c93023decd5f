"""The forms of the environment kernel's births and of the policy kernel's few
agents, with proof that each was the one that ran.

Births: the persistent kernel against the per-phase one, bit for bit, where the
phase trace shows how many claimants there were and how many barriers the step
used (3: no claimant or the fast path; 4: the general path), on the small
batch's cluster of eight CTAs and on the whole grid, for one world and for
several in a handle.  Few agents: the register variants against the ring form
on both sides of three eighths of the launch's warps, for every number of
resident warps an SM can have.  A small batch has no barrier that could be
armed to time out."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads
from tests import harness

pytestmark = pytest.mark.gpu

CLAIMANTS, BARRIERS = 11, 12        # words of a trace row
# (side, slots, founders of each world, CTAs of the persistent form, least and most claimants, barriers)
CASES = [
    (32, 60, [1], 8, 1, 1, 3),                  # cluster; single elements
    (32, 200, [20], 8, 3, 32, 3),               # cluster; runs, children merged into the list
    (64, 700, [150], 8, 33, 256, 3),            # cluster; the list's second pass again
    (128, 4096, [1500], 8, 257, 4096, 4),       # cluster; general path
    (160, 5000, [1], None, 1, 1, 3),            # grid; single elements
    (160, 5000, [30], None, 6, 32, 3),          # grid; runs
    (160, 5000, [200], None, 33, 256, 3),
    (160, 5000, [2000], None, 257, 5000, 4),
    (32, 300, [5, 80, 1], 8, 3, 256, 4),        # several worlds: the general path
    (160, 5000, [5, 1800, 40], None, 257, 5000, 4),
]


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("side,slots,founders,ctas,least,most,barriers", CASES)
def test_births(side, slots, founders, ctas, least, most, barriers, prec):
    import torch
    from paper_2510_18221_gb300 import eco
    ctas = ctas or torch.cuda.get_device_properties(0).multi_processor_count
    ws = [workloads.scaled("mid", side + 2 * e, slots, n, seed=e, precision=prec, e_init=210, wall_density=0.0, patch_k=5,
                           hidden=32) for e, n in enumerate(founders)]
    a, b = eco.Env(ws, launch_mode=0), eco.Env(ws, launch_mode=1)
    for x in (a, b):
        x.reset()
        x.prepare()
    assert a.launch_mode() == (0, ctas) and b.launch_mode()[0] == 1
    a.trace_phases(True)
    for x in (a, b):
        x.step(1)
    row = a.phase_trace()[0]
    assert least <= row[CLAIMANTS] <= most and row[BARRIERS] == barriers
    assert sum(s["births"] for s in a.stats()) >= least // 2
    for _ in range(2):
        for e in range(len(ws)):
            sa, sb = a.read_state(e), b.read_state(e)
            for k in harness.STATE_KEYS + ("colour",):
                assert np.array_equal(sa[k], sb[k]), (e, k)
            assert np.array_equal(a.read_params(e).view(np.uint32), b.read_params(e).view(np.uint32)), e
            if prec != "fp32":
                (ca, ka), (cb, kb) = a.read_streamed(e, 0, slots), b.read_streamed(e, 0, slots)
                assert np.array_equal(ca, cb) and (ka is None or np.array_equal(ka, kb)), e
                assert np.array_equal(a.read_streamed_bias(e, 0, slots), b.read_streamed_bias(e, 0, slots)), e
        assert a.stats() == b.stats() and a.stats("last") == b.stats("last")
        for x in (a, b):
            x.step(2)
    a.close()
    b.close()


@pytest.mark.parametrize("variant", [1, 2, 4, 5, 6, 9, 10])
@pytest.mark.parametrize("kw", [dict(precision="bf16"), dict(precision="fp32", patch_k=3, hidden=32),
                                dict(precision="fp8", patch_k=5, hidden=128)])
def test_few_on_both_sides_of_every_occupancy(variant, kw):
    import torch
    from paper_2510_18221_gb300 import eco
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    edges = [3 * sms * warps // 8 for warps in range(16, 52, 4)]
    top = edges[-1] + 1
    w = workloads.scaled("mid", 200, top, top, **kw)
    a, b = eco.Env(w, policy_variant=variant), eco.Env(w, policy_variant=3)
    for x in (a, b):
        x.reset()
    full = a.read_state(0)
    for n in sorted({m for e in edges for m in (e, e + 1)}, reverse=True):
        st = dict(full, alive=(np.arange(top) < n).astype(np.uint8))    # the first n slots; the others' cells stay marked
        for x in (a, b):
            x.write_state(0, {k: st[k] for k in ("alive", "x", "y")})
            x.policy_only(1)
        assert a.policy_bytes()[1] == n
        la, aa = a.read_policy_io(0)
        lb, ab = b.read_policy_io(0)
        assert np.array_equal(la.view(np.uint32), lb.view(np.uint32)) and np.array_equal(aa, ab), n
    a.close()
    b.close()


def test_a_small_batch_has_no_barrier_to_arm():
    from paper_2510_18221_gb300 import eco
    env = eco.Env(workloads.scaled("small", 64, 256, 200))
    env.reset()
    env.prepare()
    assert env.launch_mode() == (0, 8)
    with pytest.raises(eco.EcoError) as ex:
        eco.eco_arm_barrier_timeout(env.h, 0, 1000)
    assert ex.value.code == eco.ECO_EINVAL
    env.step(2)
    assert env.stats()[0]["step"] == 2
    env.close()
