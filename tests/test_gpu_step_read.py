"""eco_step_read where the environment kernel writes the host's records
itself: every step's records equal those of a handle stepped and read one
step at a time, for one world and for several (more than the warps that fold
them), in both launch forms; and a device-side wait that runs out reaches the
host through a pipelined read."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_envs,launch_mode", [(1, 0), (1, 1), (5, 0), (40, 0)])
def test_pipelined_records(n_envs, launch_mode):
    from paper_2510_18221_gb300 import eco
    ws = [workloads.scaled("mid", 32 + 4 * (e % 3), 300, 200, precision="bf16", e_init=185, seed=e) for e in range(n_envs)]
    a, b = eco.Env(ws, launch_mode=launch_mode), eco.Env(ws)
    for x in (a, b):
        x.reset()
    want = eco.eco_read_stats(b.h, n_envs)
    for t in range(7):
        got = eco.eco_step_read(a.h, n_envs)      # the records before the step it enqueues
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), t
        b.step(1)
        want = eco.eco_read_stats(b.h, n_envs)
    got = eco.eco_read_stats(a.h, n_envs)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    a.close()
    b.close()


def test_timeout_reaches_a_pipelined_read():
    from paper_2510_18221_gb300 import eco
    env = eco.Env(workloads.scaled("mid", 128, 8192, 4000, precision="bf16"))
    env.reset()
    for _ in range(3):
        eco.eco_step_read(env.h, 1)
    eco.eco_arm_barrier_timeout(env.h, env.launch_mode()[1] - 1, 100000)
    codes = []
    for _ in range(4):      # the armed step, its report, and steps that stop at once
        try:
            eco.eco_step_read(env.h, 1)
            codes.append(eco.ECO_OK)
        except eco.EcoError as ex:
            codes.append(ex.code)
    assert codes == [eco.ECO_OK] + [eco.ECO_ETIMEOUT] * 3
    env.reset()
    before = eco.eco_step_read(env.h, 1)[0][0]
    assert before[0] == 0 and eco.eco_read_stats(env.h, 1)[0][0][0] == 1
    env.close()


def test_records_of_a_step_that_timed_out():
    """The read that reports a timeout still hands over the records as the
    stopped step left them: those of the step before it."""
    from paper_2510_18221_gb300 import eco
    env = eco.Env(workloads.scaled("mid", 128, 8192, 4000, precision="bf16"))
    env.reset()
    for _ in range(3):
        eco.eco_step_read(env.h, 1)
    want = eco.eco_read_stats(env.h, 1)
    eco.eco_arm_barrier_timeout(env.h, env.launch_mode()[1] - 1, 100000)
    eco.eco_step_read(env.h, 1)
    total, last = np.zeros((2, 1, eco.ECO_N_STATS), np.int64)
    rc = eco.lib().eco_step_read(env.h, total.ctypes.data, last.ctypes.data, 1)
    assert rc == eco.ECO_ETIMEOUT
    assert np.array_equal(total, want[0]) and np.array_equal(last, want[1])
