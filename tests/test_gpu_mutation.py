"""The mutation's forms against one another, bit for bit: the persistent
kernel's single elements, its runs of inputs (FP32, BF16) and its FP8 tiles
against the tiles of the per-phase kernel, and the children's streamed copies
against those that eco_write_params derives from the same masters.  Births
from one to more than the fast path takes, on the small batch's cluster and on
the whole grid; observation sizes of every alignment of a Philox block, a
tile larger than the elements its threads keep, and several hidden layers."""
import numpy as np
import pytest

from paper_2510_18221_gb300 import workloads
from tests import harness

pytestmark = pytest.mark.gpu

SHAPES = [
    ("mid", dict()),                                    # D = 371, 3 mod 4
    ("mid", dict(patch_k=7, n_scalars=4, hidden=32)),   # D = 151
    ("mid", dict(patch_k=0, hidden=128)),               # D = 8: one run, below H
    ("mid", dict(patch_k=15, hidden=32)),               # D = 683: 8 x 683 elements a tile
    ("paperform", dict(n_hidden=3)),
    ("terrain", dict(patch_k=5)),                       # D = 116, 0 mod 4
]


def _births(key, kw, prec, side, slots, n):
    rich = dict(e_init=210) if key != "terrain" else dict(e_init=390, b_body=10)
    return workloads.scaled(key, side, slots, n, precision=prec, **rich, **kw)


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
@pytest.mark.parametrize("key,kw", SHAPES)
def test_children_alike(key, kw, prec):
    from paper_2510_18221_gb300 import eco
    for side, slots, n in ((32, 60, 1), (64, 700, 300), (160, 5000, 1), (160, 5000, 40), (160, 5000, 2000)):
        w = _births(key, kw, prec, side, slots, n)
        a, b = eco.Env(w, launch_mode=0), eco.Env(w, launch_mode=1)
        for x in (a, b):
            x.reset()
            x.step(3)
        assert a.launch_mode()[0] == 0 and b.launch_mode()[0] == 1
        sa, sb = a.read_state(0), b.read_state(0)
        for k in harness.STATE_KEYS:
            assert np.array_equal(sa[k], sb[k]), (k, side, n)
        if key != "terrain" and n > 1:      # one founder may have a wall behind it
            assert (sa["birth_step"] >= 0).any(), (side, n)
        pa, pb = a.read_params(0), b.read_params(0)
        assert np.array_equal(pa.view(np.uint32), pb.view(np.uint32)), (side, n)
        if prec != "fp32":
            (ca, ka), (cb, kb) = a.read_streamed(0, 0, slots), b.read_streamed(0, 0, slots)
            b.write_params(0, 0, pa)
            cw, kw_ = b.read_streamed(0, 0, slots)
            assert np.array_equal(ca, cb) and np.array_equal(ca, cw), (side, n)
            assert np.array_equal(a.read_streamed_bias(0, 0, slots), b.read_streamed_bias(0, 0, slots))
            if prec == "fp8":
                assert np.array_equal(ka, kb) and np.array_equal(ka, kw_), (side, n)
        a.close()
        b.close()
