"""eco_policy_bytes and eco_policy_only right after a step that timed out and
whose status nobody has read: they take the agents that the state holds, not
the list of an earlier step.  The step is stopped through
eco_arm_barrier_timeout; the state of one that stopped between its deaths and
its list is then made by clearing alive bytes in the caller's workspace."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("how", ["step", "timed", "read"])
def test_policy_takes_the_state_s_agents(how):
    import torch
    from paper_2510_18221_gb300 import eco
    env = eco.Env(workloads.scaled("mid", 128, 8192, 4000, precision="bf16", e_init=190))
    env.reset()
    env.step(3)
    assert env.policy_bytes()[1] == env.stats()[0]["alive"]
    eco.eco_arm_barrier_timeout(env.h, env.launch_mode()[1] - 1, 100000)
    {"step": lambda: env.step(1), "timed": lambda: env.step_timed(1), "read": lambda: eco.eco_step_read(env.h, 1)}[how]()
    env.stream.synchronize()
    alive = env.read_state(0)["alive"]
    logits = env.read_policy_io(0)[0]
    # the alive bytes in the workspace: the first place with this pattern (the
    # region that state reads pass through, which holds a copy, comes last)
    at = env.workspace.cpu().numpy().tobytes().find(alive.tobytes())
    assert at >= 0
    gone = np.flatnonzero(alive)[::7]
    alive[gone] = 0
    env.workspace[at:at + len(alive)] = torch.from_numpy(alive).cuda()
    torch.cuda.synchronize()
    env.policy_only(1)
    assert env.policy_bytes()[1] == int(alive.sum())
    after = env.read_policy_io(0)[0]
    assert np.array_equal(after[gone].view(np.uint32), logits[gone].view(np.uint32))
    moved = (after != logits).any(axis=1)
    assert moved[alive.astype(bool)].mean() > 0.5      # the step's moves are in: another observation
    with pytest.raises(eco.EcoError) as ex:
        env.stats()
    assert ex.value.code == eco.ECO_ETIMEOUT
    env.reset()
    assert env.policy_bytes()[1] == 4000
    env.close()
