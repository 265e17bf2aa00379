"""2D level updates that take their rebuilt and TN nodes along.

A run with few such nodes spreads each over several lanes, a large batch takes
one lane per node; the sums are formed in the same order, so a run gives the
same bits alone (many lanes) and in a batch past the crossover (one lane).
Against the oracle: the parity bound of the other binary32 tests, 1e-6, on
layouts whose faces are not a multiple of a warp, boxes with corners, slabs
without, a box that touches the periodic seam, and three levels.
"""
import numpy as np
import pytest

from paper_2004_11863_gb300 import workloads as W

pytestmark = pytest.mark.gpu

IC = dict(kind="random", seed=11, u0=(0.05, -0.03, 0.0), drho=1e-3, du=5e-3)
REST = dict(kind="random", seed=12, drho=1e-3, du=5e-3)
LAYOUTS = {
    "box": ((33, 29, 1), [((8, 7, 0), (24, 20, 1))]),
    "slab_x": ((32, 13, 1), [((16, 0, 0), (32, 13, 1))]),   # touches the seam at x = 32
    "slab_y": ((13, 32, 1), [((0, 5, 0), (13, 20, 1))]),
    "smallest": ((8, 8, 1), [((2, 3, 0), (6, 7, 1))]),
    "nested": ((40, 36, 1), [((8, 6, 0), (32, 30, 1)), ((9, 8, 0), (38, 40, 1))]),
}


def case_of(layout, collision, ic, steps):
    dims, boxes = LAYOUTS[layout]
    return W.Case("edges_" + layout, "D2Q9", collision, 0.53, dims, boxes, ic, steps)


@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("collision,ic", [("RR", IC), ("RR", REST), ("REG", IC), ("BGK", IC)])
def test_special_nodes_match_the_oracle(layout, collision, ic):
    import oracle
    from paper_2004_11863_gb300 import mlbm

    case = case_of(layout, collision, ic, 7)
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


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("layout", ["box", "slab_x", "nested"])
def test_lanes_per_node_change_no_bit(layout, storage):
    from paper_2004_11863_gb300 import mlbm

    # 4 lanes an outer node, 16 a TN node: past 65,536 lanes at 200 runs on
    # every level that has such nodes
    case = case_of(layout, "RR", IC, 6)
    alone = mlbm.Lbm.from_case(case, storage=storage)
    batch = mlbm.Lbm.from_case(case, storage=storage, batch=200)
    alone.step(6)
    batch.step(6)
    for l in range(case.nlevels):
        want = alone.populations(l)
        for b in (0, 1, 198, 199):
            assert np.array_equal(batch.populations(l, run=b), want)
    alone.close()
    batch.close()


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q19"])
def test_six_step_graphs_match_single_launches(lattice):
    """Calls that cross, fill and miss the six-step period, with probes."""
    from paper_2004_11863_gb300 import mlbm

    case = W.small_2level_2d("RR") if lattice == "D2Q9" else W.small_3d("D3Q19", "RR", 2)
    runs = []
    for graphs in (True, False):
        g = mlbm.Lbm.from_case(case)
        g.set_graphs(graphs)
        g.probe_add(1, [[3, 3, 0], [5, 4, 0]])
        for n in (1, 13, 20, 6, 7, 12, 5):
            g.step(n)
        runs.append((g.probe(), [g.populations(l) for l in range(2)]))
        g.close()
    assert runs[0][0].shape[0] == 64 and np.array_equal(runs[0][0], runs[1][0])
    for l in range(2):
        assert np.array_equal(runs[0][1][l], runs[1][1][l])
