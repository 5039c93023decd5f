"""The workspace region that eco_read_state converts arrays in: it holds a
world's cells and slots (a small world's whole state) also where the slots'
parameters alone would need far less, so that a large world of few agents is
read in one piece.  Seen through eco_workspace_bytes on the CPU; the states
themselves, in one piece and in several, against the oracle on the GPU."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads

# bytes that a cell takes in the workspace's arrays: flags 1, occupant 4, move
# claim 8 and count 4, birth claim 8, attack 8, energy, rock, water, biomass,
# photosynthesis remainder and flow 4 each
CELL_BYTES = 57
REGION = 32 << 20


def _world(side, slots):
    return workloads.scaled("small", side, slots, min(slots, 3), patch_k=3, hidden=32)


def _bytes(side, slots):
    from paper_2510_18221_gb300 import eco
    cfg, keep = eco.make_config([_world(side, slots)])
    return eco.eco_workspace_bytes(cfg)


@pytest.mark.parametrize("side,slots", [(256, 1), (1024, 4), (2048, 64), (4096, 2)])
def test_region_holds_the_cells(side, slots):
    small = _bytes(32, slots)
    cells = side * side - 32 * 32
    staged = _bytes(side, slots) - small - CELL_BYTES * cells
    # every region is rounded up to 256 bytes; the small world's own region
    # (its whole state, at most 32 KB + 50 bytes a slot, or the parameters)
    assert staged >= min(6 * side * side, REGION) - (64 << 10) - 10000 * slots
    assert staged <= REGION + (64 << 10)


@pytest.mark.gpu
@pytest.mark.parametrize("side,slots", [(30, 1), (200, 2), (218, 2), (220, 3), (1024, 4), (2400, 5)])    # 2400: two pieces
def test_few_slots_many_cells(side, slots):
    import oracle
    from paper_2510_18221_gb300 import eco
    from tests import harness
    w = _world(side, slots)
    env, orc = eco.Env(w), oracle.Oracle(w)
    env.reset()
    orc.reset()
    got = env.read_state(0)
    harness.compare_state(got, orc, "side %d" % side)
    assert np.array_equal(got["colour"], orc.colour)
    env.close()
