"""State and parameters of one handle read and written by several host
threads at once: each gets what it asked for, although the transfers share the
workspace's staging region and one pinned buffer.  Worlds that are read
through the pinned buffer and one that is read in pieces; parameter runs of
one chunk and of several."""
import threading

import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads

pytestmark = pytest.mark.gpu


def _all(works):
    errors = []

    def guard(i, f):
        try:
            f()
        except Exception as ex:     # noqa: BLE001 -- reported by the main thread
            errors.append("%d: %s" % (i, ex))

    threads = [threading.Thread(target=guard, args=(i, f)) for i, f in enumerate(works)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


@pytest.mark.parametrize("prec", ["fp32", "fp8"])
def test_threads_share_a_handle(prec):
    from paper_2510_18221_gb300 import eco
    ws = [workloads.scaled("mid", side, slots, n, precision=prec, seed=i)
          for i, (side, slots, n) in enumerate([(32, 60, 40), (30, 70, 50), (640, 600, 500)])]
    env = eco.Env(ws)
    env.reset()
    states = [env.read_state(e) for e in range(3)]
    params = [env.read_params(e) for e in range(3)]
    again = np.random.default_rng(0).standard_normal((40, env.P)).astype(np.float32)

    def read_state(e, n):
        for _ in range(n):
            got = env.read_state(e)
            for k, want in states[e].items():
                assert np.array_equal(got[k], want), (e, k)

    def read_params(e, slot0, count, n):
        for _ in range(n):
            got = env.read_params(e, slot0, count)
            assert np.array_equal(got.view(np.uint32), params[e][slot0:slot0 + count].view(np.uint32)), (e, slot0)

    def write_params(n):            # slots that nobody else reads
        for _ in range(n):
            env.write_params(2, 560, again)
            assert np.array_equal(env.read_params(2, 560, 40).view(np.uint32), again.view(np.uint32))

    assert _all([lambda: read_state(0, 60), lambda: read_state(1, 60), lambda: read_state(2, 10),
                 lambda: read_params(0, 0, 60, 40), lambda: read_params(2, 0, 200, 20), lambda: read_params(2, 200, 360, 10),
                 lambda: write_params(20)]) == []
    env.close()
