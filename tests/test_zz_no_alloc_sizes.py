"""eco_move_claims_noalloc on both sides of its one-launch limit (16,384
agents), at the edges of its CTAs and of its agents per thread, against the
rule itself in numpy with the oracle's Philox draws; two calls in a row, the
second over the first one's scratch."""
import numpy as np
import pytest

import oracle
from paper_2510_18221_gb300 import eco

pytestmark = pytest.mark.gpu

DX, DY = np.array([0, 1, 0, -1]), np.array([-1, 0, 1, 0])
FACE = {1: 0, 2: 2, 3: 1, 4: 3}


def _rule(side, pos, act, fac, blocked, seed, step):
    face, new, moved, best = fac.copy(), pos.copy(), np.zeros(len(pos), np.uint8), {}
    for i, a in enumerate(act):
        if a in FACE:
            face[i] = FACE[a]
            x, y = (pos[i] % side + DX[face[i]]) % side, (pos[i] // side + DY[face[i]]) % side
            c = int(y * side + x)
            if 0 <= pos[i] < side * side and not blocked[c]:
                best[c] = max(best.get(c, (-1, 0)), (oracle.philox((step, i, 0, 0), (seed, 7))[0], -i))
        elif a in (6, 7):
            face[i] = (face[i] + (3 if a == 6 else 1)) & 3
    for c, (_, neg) in best.items():
        new[-neg], moved[-neg] = c, 1
    return face, new, moved


@pytest.mark.parametrize("side,n", [(4, 1), (6, 30), (64, 1023), (200, 8192), (200, 8193), (512, 16384), (512, 16385)])
def test_claims_match_the_rule(side, n):
    import torch
    rng = np.random.default_rng(n)
    for call in range(2):
        pos = rng.choice(side * side, size=n, replace=False).astype(np.int32)
        blocked = (rng.random(side * side) < 0.02).astype(np.uint8)
        blocked[pos] = 1
        act, fac = rng.integers(0, 9, n).astype(np.uint8), rng.integers(0, 4, n).astype(np.uint8)
        if n > 20:
            pos[3] = -1                       # outside the grid: turns, does not move
            pos[4] = side * side
        dev = [torch.from_numpy(a).cuda() for a in (pos, act, fac, blocked)]
        out = [torch.empty(n, dtype=t, device="cuda") for t in (torch.uint8, torch.int32, torch.uint8)]
        torch.cuda.synchronize()
        eco.eco_move_claims_noalloc(side, n, dev[0].data_ptr(), dev[1].data_ptr(), dev[2].data_ptr(), dev[3].data_ptr(),
                                    5, 11 + call, out[0].data_ptr(), out[1].data_ptr(), out[2].data_ptr(), 0)
        torch.cuda.synchronize()
        for got, want in zip(out, _rule(side, pos.astype(np.int64), act, fac, blocked, 5, 11 + call)):
            assert np.array_equal(got.cpu().numpy(), want), call
