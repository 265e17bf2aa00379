"""The even binary16 3D update that moves two neighbours per access, for every
collision and with the reference at rest and moving (an instance, and for BGK a
launch bound, of its own each): the bits of the same runs in pairs, which
another kernel updates, on rows with an odd end, odd numbers of rows, ghost
nodes, faces normal to x and inactive nodes beside them."""
import numpy as np
import pytest

from paper_2004_11863_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MOVING = dict(kind="random", seed=41, u0=(0.04, -0.02, 0.03), drho=1e-3, du=5e-3)
REST = dict(kind="random", seed=42, drho=1e-3, du=5e-3)
LAYOUTS = {
    "short": ((4, 5, 4), []),
    "row33": ((33, 7, 6), []),
    "box": ((17, 15, 14), [((4, 4, 4), (12, 11, 9))]),
    "seam_x": ((20, 9, 8), [((10, 0, 0), (20, 9, 8))]),
    "walls_yz": ((34, 13, 12), [((0, 4, 3), (34, 9, 8))]),
}


@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("lattice", ["D3Q19", "D3Q27"])
@pytest.mark.parametrize("collision,ic", [("BGK", MOVING), ("BGK", REST), ("REG", MOVING),
                                          ("REG", REST), ("RR", REST)])
def test_alone_and_in_pairs(layout, lattice, collision, ic):
    from paper_2004_11863_gb300 import mlbm

    dims, boxes = LAYOUTS[layout]
    case = W.Case("half", lattice, collision, 0.54, dims, boxes, ic, 5)
    alone = mlbm.Lbm.from_case(case, storage="fp16")
    pairs = mlbm.Lbm.from_case(case, storage="fp16", batch=2)
    alone.step(5)
    pairs.step(5)
    for l in range(case.nlevels):
        want = alone.populations(l)
        assert np.any(want)
        for b in range(2):
            assert np.array_equal(pairs.populations(l, run=b), want)
    alone.close()
    pairs.close()
