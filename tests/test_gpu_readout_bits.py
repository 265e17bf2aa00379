"""The binary32 read-out is the FP64 one rounded once, bit for bit: over flows
whose values sit on and beside the halfway points of binary32 (a uniform far
field), cancel the reference's momentum (a flow at rest under a moving
reference), run down to subnormal numbers (the tails of a pulse at rest) or
have a density far from one."""
import numpy as np
import pytest

from paper_2004_11863_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LAYOUT = {"D2Q9": ((160, 96, 1), [((80, 0, 0), (160, 96, 1))]),
          "D3Q19": ((48, 40, 33), [((14, 10, 9), (34, 28, 25))]),
          "D3Q27": ((40, 36, 30), [((11, 10, 9), (30, 26, 22))])}


def check(h):
    import torch

    for l in range(h.nlevels):
        n = h.nodes(l)
        for b in range(h.batch):
            rho = torch.full((n,), 7.0, device="cuda")
            u = torch.full((3, n), 7.0, device="cuda")
            torch.cuda.synchronize()
            h.macros_device(l, rho.data_ptr(), u.data_ptr(), run=b)
            h.sync()
            with np.errstate(over="ignore"):
                want = [x.astype(np.float32) for x in h.macros(l, run=b)]
            for got, w in zip((rho.cpu().numpy(), u.cpu().numpy()), want):
                assert np.array_equal(got, w, equal_nan=True)


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("lattice", LAYOUT)
@pytest.mark.parametrize("kind,u0,u_ref,rho0", [
    ("vortex", 0.1, 0.1, 1.0),
    ("vortex", 0.07, 0.07, 1.2),
    ("pulse", 0.0, 0.0, 1.0),
    ("pulse", 0.0, 0.06, 1.0),      # cancels rho0 U nearly everywhere
    ("uniform", 0.0, 0.06, 1.0),
    ("pulse", 0.05, 0.0, 1000.0),
    ("pulse", 0.05, 0.05, 1e-3),
    ("pulse", 0.05, 0.05, 3e-25),   # the whole field by way of FP64
])
def test_rounded_once(lattice, storage, kind, u0, u_ref, rho0):
    from paper_2004_11863_gb300 import mlbm

    if storage == "fp16" and rho0 < 1e-2:
        pytest.skip("populations below the range of binary16")
    dims, boxes = LAYOUT[lattice]
    h = mlbm.Lbm(lattice, "RR", 0.51, dims, boxes, storage=storage, batch=2, rho0=rho0,
                 u_ref=(u_ref, 0.0, 0.0))
    for b in range(2):
        h.init_analytic(dict(kind=kind, u0=(u0, 0.0, 0.0),
                             center=(dims[0] * 0.4 + b, dims[1] * 0.5,
                                     dims[2] * 0.5 if lattice != "D2Q9" else 0.0),
                             radius=3.0, amplitude=1e-3 * rho0, eps=0.03, drho=0.0), b)
    check(h)
    for n in (1, 6, 20):
        h.step(n)
        check(h)
    h.close()


@pytest.mark.parametrize("lattice", LAYOUT)
def test_random_fields(lattice):
    from paper_2004_11863_gb300 import mlbm

    dims, boxes = LAYOUT[lattice]
    case = W.Case("bits", lattice, "RR", 0.55, dims, boxes,
                  dict(kind="random", seed=5, u0=(0.03, 0.0, 0.0), drho=1e-2, du=3e-2), 3)
    h = mlbm.Lbm.from_case(case)
    check(h)
    h.step(3)
    check(h)
    h.close()
