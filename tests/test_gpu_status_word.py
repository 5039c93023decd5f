"""The status word of the host's copy of a step (eco_step_read): the step stores
it only when it is not 0, so both copies report a timeout on every call until a
reset, and neither keeps it behind the reset; a reset that found too few cells
is reported by every read of its steps too."""
import pytest

from paper_2510_18221_gb300 import workloads

pytestmark = pytest.mark.gpu


def _codes(eco, env, n):
    out = []
    for _ in range(n):
        try:
            eco.eco_step_read(env.h, env.n_envs)
            out.append(eco.ECO_OK)
        except eco.EcoError as ex:
            out.append(ex.code)
    return out


@pytest.mark.parametrize("before", [0, 1, 2])       # calls before the armed one: either copy comes first
def test_timeout_in_both_copies_until_a_reset(before):
    from paper_2510_18221_gb300 import eco
    env = eco.Env(workloads.scaled("mid", 128, 8192, 4000, precision="bf16"))
    env.reset()
    env.prepare()
    assert _codes(eco, env, before) == [eco.ECO_OK] * before
    eco.eco_arm_barrier_timeout(env.h, env.launch_mode()[1] - 1, 100000)
    assert _codes(eco, env, 6) == [eco.ECO_OK] + [eco.ECO_ETIMEOUT] * 5
    env.reset()
    assert _codes(eco, env, 6) == [eco.ECO_OK] * 6
    assert eco.eco_read_stats(env.h, 1)[0][0][0] == 6
    env.close()


@pytest.mark.parametrize("side,slots,launch_mode", [(32, 900, 0), (32, 900, 1), (160, 25000, 0)])
def test_failed_reset_in_every_read(side, slots, launch_mode):
    from paper_2510_18221_gb300 import eco
    env = eco.Env(workloads.scaled("mid", side, slots, slots, precision="bf16", wall_density=0.5, patch_k=3, hidden=32),
                  launch_mode=launch_mode)
    with pytest.raises(eco.EcoError) as ex:
        env.reset()
    assert ex.value.code == eco.ECO_EINVAL
    assert _codes(eco, env, 5) == [eco.ECO_EINVAL] * 5
    env.close()
