"""Read-outs queued behind one another (their launches overlap), between steps
and copies, without a wait in between: the bits of a run that waits after every
call.  Also recorded into a CUDA graph and replayed."""
import pytest

from paper_2004_11863_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BOX = {"D2Q9": ((96, 64, 1), [((24, 16, 0), (72, 48, 1))]),
       "D3Q19": ((24, 20, 16), [((6, 5, 4), (18, 15, 12))]),
       "D3Q27": ((20, 16, 16), [((5, 4, 4), (15, 12, 12))])}


def opened(lattice, storage, batch, stream):
    from paper_2004_11863_gb300 import mlbm

    dims, boxes = BOX[lattice]
    h = mlbm.Lbm(lattice, "RR", 0.55, dims, boxes, storage=storage, batch=batch, stream=stream)
    for b in range(batch):
        h.init_analytic(dict(kind="pulse", center=(dims[0] * 0.3 + b, dims[1] * 0.5, dims[2] * 0.5),
                             radius=3.0, amplitude=1e-2), b)
    return h


def buffers(h):
    import torch
    return [(torch.zeros(h.batch, h.nodes(l), device="cuda"),
             torch.zeros(h.batch, 3, h.nodes(l), device="cuda")) for l in range(h.nlevels)]


def read(h, out, wait=False):
    for l, (rho, u) in enumerate(out):
        for b in range(h.batch):
            h.macros_device(l, rho[b].data_ptr(), u[b].data_ptr(), run=b)
            if wait:
                h.sync()


def same(a, b):
    import torch
    return all(torch.equal(torch.nan_to_num(x, nan=-7.0), torch.nan_to_num(y, nan=-7.0))
               for p, q in zip(a, b) for x, y in zip(p, q))


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("lattice", BOX)
def test_queued_reads(lattice, storage):
    import torch

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = opened(lattice, storage, 7, s.cuda_stream)
        out = buffers(h)
        first, second = buffers(h), buffers(h)
        keep = lambda to: [x.copy_(y, non_blocking=True)  # noqa: E731
                           for p, q in zip(to, out) for x, y in zip(p, q)]
        torch.cuda.synchronize()
        h.step(4)
        read(h, out)
        keep(first)
        h.step(7)
        read(h, out)
        h.step(1)
        read(h, out)
        keep(second)
        torch.cuda.synchronize()
        w = opened(lattice, storage, 7, s.cuda_stream)
        a, b = buffers(w), buffers(w)
        torch.cuda.synchronize()
        for n, to in ((4, a), (8, b)):
            for _ in range(n):
                w.step(1)
                w.sync()
            read(w, to, wait=True)
        torch.cuda.synchronize()
        assert same(first, a) and same(second, b)
        assert not same(first, second)
    h.close()
    w.close()


@pytest.mark.parametrize("lattice", BOX)
def test_reads_in_a_captured_graph(lattice):
    import torch

    s = torch.cuda.Stream()
    h = opened(lattice, "fp32", 3, s.cuda_stream)
    out, want = buffers(h), buffers(h)
    h.step(3)
    read(h, want, wait=True)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        read(h, out)
        doubled = [(rho * 2.0, u * 2.0) for rho, u in out]
    for _ in range(3):
        for p in out:
            for x in p:
                x.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            g.replay()
        torch.cuda.synchronize()
        assert same(out, want)
        assert same(doubled, [(rho * 2.0, u * 2.0) for rho, u in want])
    del g
    h.close()
