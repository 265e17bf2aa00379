"""The binary32 read-out (lbm_macros_device) against the FP64 one (lbm_macros).

Both form the sums of the populations to FP64 accuracy; the binary32 one then
rounds once, so the two agree to one unit in the last binary32 place (2^-23
relative) plus the summation bound of both (1e-12 of values of order one),
and both give NaN at the inactive nodes.
"""
import numpy as np
import pytest

from paper_2004_11863_gb300 import workloads as W

pytestmark = pytest.mark.gpu

U = (0.05, -0.02, 0.01)


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("lattice,dims,levels,batch,u0", [
    ("D2Q9", (33, 4, 1), 1, 1, (0.0, 0.0, 0.0)),       # one node past a warp; the smallest rows
    ("D2Q9", (96, 64, 1), 2, 3, U[:2] + (0.0,)),       # inactive nodes, several runs
    ("D3Q19", (24, 20, 16), 2, 1, U),
    ("D3Q27", (31, 17, 9), 1, 2, U),
    ("D3Q27", (24, 20, 16), 2, 1, (0.0, 0.0, 0.0)),
])
def test_binary32_readout_rounds_the_fp64_one(lattice, dims, levels, batch, u0, storage):
    import torch

    from paper_2004_11863_gb300 import mlbm

    boxes = []
    if levels == 2:
        boxes = [((24, 16, 0), (72, 48, 1))] if lattice == "D2Q9" else [((6, 5, 4), (18, 15, 12))]
    case = W.Case("readout", lattice, "RR", 0.55, dims, boxes,
                  dict(kind="random", seed=3, u0=u0, drho=1e-2, du=2e-2), 3)
    h = mlbm.Lbm.from_case(case, storage=storage, batch=batch)
    h.step(3)
    for l in range(levels):
        n = h.nodes(l)
        for b in range(batch):
            rho = torch.zeros(n, device="cuda")
            u = torch.zeros(3, n, device="cuda")
            torch.cuda.synchronize()
            h.macros_device(l, rho.data_ptr(), u.data_ptr(), run=b)
            h.sync()
            r64, u64 = h.macros(l, run=b)
            for got, want in ((rho.cpu().numpy(), r64), (u.cpu().numpy(), u64)):
                assert np.array_equal(np.isnan(got), np.isnan(want))
                ok = ~np.isnan(want)
                err = np.abs(got.astype(np.float64)[ok] - want[ok])
                assert np.all(err <= 2.0 ** -23 * np.abs(want[ok]) + 2e-12)
    h.close()
