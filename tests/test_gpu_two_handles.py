"""Two live handles of different shapes: the shared-memory limit of a kernel
belongs to the function, so a handle with a smaller observation, created or
driven in between, leaves the larger one everything it could do -- policy
passes, the first step (whose graphs are captured then), reset, parameter I/O --
with the results it has alone; also from two host threads at once."""
import threading

import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads
from tests import harness

pytestmark = pytest.mark.gpu


def _world(k, prec, n=900):
    return workloads.scaled("mid", 96, n + 100, n, precision=prec, patch_k=k, e_init=190)


def _outputs(env):
    return [env.read_state(0)[k] for k in harness.STATE_KEYS] + [a.view(np.uint8) for a in env.read_policy_io(0)] + \
        [env.read_params(0).view(np.uint32)]


@pytest.mark.parametrize("launch_mode", [0, 1])
@pytest.mark.parametrize("prec,variant", [("fp32", 6), ("bf16", 3), ("fp8", 8)])
def test_smaller_handle_between(prec, variant, launch_mode):
    from paper_2510_18221_gb300 import eco
    def make(k):
        return eco.Env(_world(k, prec), policy_variant=variant, launch_mode=launch_mode)
    alone = make(15)
    alone.reset()
    alone.policy_only(1)
    alone.step(2)
    want = _outputs(alone)
    alone.close()
    big = make(15)
    big.reset()
    small = make(3)
    small.reset()
    big.policy_only(1)
    small.step(1)
    big.step(2)             # captures its graphs now
    small.write_params(0, 0, small.read_params(0, 0, 3))
    assert big.launch_mode()[0] == launch_mode
    got = _outputs(big)
    assert all(np.array_equal(g, w) for g, w in zip(got, want))
    big.write_params(0, 0, big.read_params(0))
    small.reset()
    big.reset()
    big.policy_only(1)
    big.step(2)
    assert all(np.array_equal(g, w) for g, w in zip(_outputs(big), want))
    big.close()
    small.close()


def test_two_threads_two_shapes():
    from paper_2510_18221_gb300 import eco
    envs = [eco.Env(_world(k, "bf16", 300), policy_variant=6) for k in (15, 3)]
    for env in envs:
        env.reset()
    want, errors = [env.read_params(0) for env in envs], []

    def work(i):
        try:
            for _ in range(40):
                envs[i].reset()
                got = envs[i].read_params(0)
                envs[i].write_params(0, 0, got)
                if not np.array_equal(got.view(np.uint32), want[i].view(np.uint32)):
                    raise AssertionError("other parameters")
        except Exception as ex:     # noqa: BLE001 -- reported by the main thread
            errors.append("%d: %s" % (i, ex))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert errors == []
    for env in envs:
        env.close()
