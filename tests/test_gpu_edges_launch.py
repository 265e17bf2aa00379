"""Special nodes of 2D levels in a launch of their own: large batches (one lane
a node) and levels with sensors.

The batch is large enough for every level that has such nodes (more than 65,536
lanes, four an outer node and sixteen a TN node, asserted): its last run gives
the bits of the run alone, which takes them within the update's launch, and
agrees with the oracle to the 1e-6 of the other binary32 tests.  Sensors only
look: with them on any set of levels a run gives the same bits, alone and in a
batch, the sensors' own values are the same in both, and no node is rebuilt
twice.
"""
import numpy as np
import pytest

from paper_2004_11863_gb300 import workloads as W

pytestmark = pytest.mark.gpu

IC = dict(kind="random", seed=31, u0=(0.05, -0.03, 0.0), drho=1e-3, du=5e-3)
REST = dict(kind="random", seed=32, drho=1e-3, du=5e-3)
LAYOUTS = {
    "box": ((33, 29, 1), [((8, 7, 0), (24, 20, 1))]),
    "slab_x": ((32, 13, 1), [((16, 0, 0), (32, 13, 1))]),   # periodic tangents: the
    "slab_y": ((13, 32, 1), [((0, 5, 0), (13, 20, 1))]),    # stencil wraps at the seam
    "smallest": ((8, 8, 1), [((2, 3, 0), (6, 7, 1))]),
    "nested": ((40, 36, 1), [((8, 6, 0), (32, 30, 1)), ((9, 8, 0), (38, 40, 1))]),
}


def case_of(layout, collision="RR", ic=IC):
    dims, boxes = LAYOUTS[layout]
    return W.Case("edges_" + layout, "D2Q9", collision, 0.53, dims, boxes, ic, 5)


def lanes(layout):
    """Lanes of the special nodes of each level's update, one run."""
    dims, boxes = LAYOUTS[layout]
    n, per = list(dims[:2]), [True, True]
    out = [0] * (len(boxes) + 1)
    for l, (lo, hi) in enumerate(boxes):
        E = [hi[a] - lo[a] for a in range(2)]
        whole = [per[a] and E[a] == n[a] for a in range(2)]
        m = [2 * n[a] if whole[a] else 2 * E[a] + 1 for a in range(2)]
        inner = lambda k, cut: np.prod([k[a] if whole[a] else k[a] - cut for a in range(2)])
        out[l] += 16 * int(inner([n[a] if whole[a] else E[a] - 1 for a in range(2)], 0)
                           - inner([n[a] if whole[a] else E[a] - 1 for a in range(2)], 2))
        out[l + 1] += 4 * int(np.prod(m) - inner(m, 2))
        n, per = m, [per[a] and whole[a] for a in range(2)]
    return out


def batch_of(layout):
    return 65536 // min(k for k in lanes(layout) if k) + 1


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("layout", LAYOUTS)
@pytest.mark.parametrize("collision,ic", [("RR", IC), ("RR", REST), ("REG", IC), ("BGK", REST)])
def test_large_batches(layout, collision, ic, storage):
    import oracle
    from paper_2004_11863_gb300 import mlbm

    case, B = case_of(layout, collision, ic), batch_of(layout)
    assert all(k * B > 65536 for k in lanes(layout) if k)
    assert all(k <= 65536 for k in lanes(layout))
    alone = mlbm.Lbm.from_case(case, storage=storage)
    batch = mlbm.Lbm.from_case(case, storage=storage, batch=B)
    alone.step(5)
    batch.step(5)
    o = oracle.Run.from_case(case)
    o.step(5)
    for l in range(case.nlevels):
        want = alone.populations(l)
        for b in (0, B // 2, B - 1):
            assert np.array_equal(batch.populations(l, run=b), want)
        if storage == "fp32":
            rg, ug = batch.macros(l, run=B - 1)
            ro, uo = o.macros(l)
            assert np.array_equal(np.isnan(rg), np.isnan(ro))
            m = ~np.isnan(ro)
            assert np.max(np.abs(rg[m] - ro[m])) <= 1e-6
            assert np.max(np.abs(ug[:, m] - uo[:, m])) <= 1e-6
    for r in (alone, batch, o):
        r.close()


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("layout,levels", [("box", (0,)), ("box", (1,)), ("slab_y", (0, 1)),
                                           ("nested", (1,)), ("nested", (0, 2)),
                                           ("nested", (0, 1, 2))])
def test_sensors_change_no_bit(layout, levels, storage):
    from paper_2004_11863_gb300 import mlbm

    case, B = case_of(layout), batch_of(layout)
    plain = mlbm.Lbm.from_case(case, storage=storage)
    alone = mlbm.Lbm.from_case(case, storage=storage)
    batch = mlbm.Lbm.from_case(case, storage=storage, batch=B)
    for r in (alone, batch):
        for l in levels:
            r.sensors_enable(l, 5e-7, 1e-6)
    for r in (plain, alone, batch):
        r.step(4)
        r.step(9)
    for l in range(case.nlevels):
        want = plain.populations(l)
        assert np.array_equal(alone.populations(l), want)
        assert np.array_equal(batch.populations(l, run=B - 1), want)
    for l in levels:
        for a, b in zip(alone.sensors(l, with_gnorm=True),
                        batch.sensors(l, run=B - 1, with_gnorm=True)):
            assert np.array_equal(a, b)
    for r in (plain, alone, batch):
        r.close()


def test_sensors_rebuild_no_node_twice():
    """A coarse step of two levels is a capture and three updates; sensors on
    level 0 add its special nodes, a velocity pass and the sensors."""
    from paper_2004_11863_gb300 import mlbm

    for levels, more in (((), 0), ((0,), 3), ((1,), 6), ((0, 1), 9)):
        r = mlbm.Lbm.from_case(case_of("box"))
        for l in levels:
            r.sensors_enable(l, 5e-7, 1e-6)
        r.step(1)
        before = r.kernel_launches()
        r.step(1)
        assert r.kernel_launches() - before == 4 + more
        r.close()
