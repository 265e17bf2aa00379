"""3D updates whose warps run along the elements of a plane.

Row lengths at which a warp holds the end of one row and the start of the
next, an odd number of rows (the last row has no partner), levels without
padding, with ghost nodes and with faces normal to x, several runs: against
the oracle within 1e-6 (binary32), and binary16 runs alone and in pairs bit
for bit.
"""
import numpy as np
import pytest

from paper_2004_11863_gb300 import workloads as W

pytestmark = pytest.mark.gpu

IC = dict(kind="random", seed=21, u0=(0.04, -0.02, 0.03), drho=1e-3, du=5e-3)
LAYOUTS = {
    "short": ((4, 5, 4), []),
    "row33": ((33, 7, 6), []),
    "row63": ((63, 4, 5), []),
    "box": ((17, 15, 14), [((4, 4, 4), (12, 11, 9))]),      # 17 x 15 x 11 inside
    "seam_x": ((20, 9, 8), [((10, 0, 0), (20, 9, 8))]),     # 21 x 18 x 16, touches x = 20
    "walls_yz": ((34, 13, 12), [((0, 4, 3), (34, 9, 8))]),  # 68 x 11 x 11, x periodic
}


@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("lattice,collision", [("D3Q19", "RR"), ("D3Q27", "RR"), ("D3Q27", "BGK"),
                                               ("D3Q19", "HRR")])
def test_rows_match_the_oracle(layout, lattice, collision):
    import oracle
    from paper_2004_11863_gb300 import mlbm

    dims, boxes = LAYOUTS[layout]
    case = W.Case("planes", lattice, collision, 0.54, dims, boxes, IC, 5)
    g = mlbm.Lbm.from_case(case)
    g.step(case.steps)
    o = oracle.Run.from_case(case)
    o.step(case.steps)
    for l in range(case.nlevels):
        rg, ug = g.macros(l)
        ro, uo = o.macros(l)
        assert np.array_equal(np.isnan(rg), np.isnan(ro))
        m = ~np.isnan(ro)
        assert np.max(np.abs(rg[m] - ro[m])) <= 1e-6
        assert np.max(np.abs(ug[:, m] - uo[:, m])) <= 1e-6
    g.close()
    o.close()


@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("lattice", ["D3Q19", "D3Q27"])
def test_binary16_alone_and_in_pairs(layout, lattice):
    from paper_2004_11863_gb300 import mlbm

    dims, boxes = LAYOUTS[layout]
    case = W.Case("planes", lattice, "RR", 0.54, dims, boxes, IC, 5)
    alone = mlbm.Lbm.from_case(case, storage="fp16")
    pairs = mlbm.Lbm.from_case(case, storage="fp16", batch=3)
    alone.step(5)
    pairs.step(5)
    for l in range(case.nlevels):
        want = alone.populations(l)
        for b in range(3):
            assert np.array_equal(pairs.populations(l, run=b), want)
    alone.close()
    pairs.close()
