"""Performance cases of the multi-level lattice Boltzmann step.

A case is one run (or a batch of runs sharing a layout) advanced by a few
coarse steps, after which the density and velocity of every level of every
run are read out on the device -- the loop of a program that uses this
library: ``step`` a chunk, ``macros_device``, look, go on.  The ranges are
those of the library's own workloads: the 2D and 3D configurations of the
benchmark, the sizes of its serving stream (2D coarse sides 64-1024, 3D
48-160, one to three levels, Mach 0.05-0.2, tau - 1/2 from 1e-5 to 1e-2) and
batches up to the benchmark's 33 runs; every lattice, collision and storage.

Keys of a case: lattice, collision, storage, nx, ny, nz (level-0 nodes),
levels, slab (the refined level spans y and z and the upper half of x;
otherwise every box is the central half of its parent), batch, steps (coarse
steps of a pass), dtau (tau_0 - 1/2), ma (Mach number of the mean flow along
x, which is also the reference velocity), ic (pulse or vortex), size (radius
of the pulse or vortex), request (the pass also creates, initialises and
closes the run, as the server does for a short request).
"""
import math
import random

import torch

from paper_2004_11863_gb300 import mlbm

CS = 1.0 / math.sqrt(3.0)
Q = {"D2Q9": 9, "D3Q19": 19, "D3Q27": 27}
SIGMA = 0.995  # the hybrid weight of the paper's runs


def _case(name, lattice, collision, dims, levels, steps, **kw):
    c = dict(name=name, lattice=lattice, collision=collision, storage="fp32", nx=dims[0],
             ny=dims[1], nz=dims[2] if len(dims) > 2 else 1, levels=levels, slab=False, batch=1,
             steps=steps, dtau=1e-4, ma=0.1, ic="vortex", size=6.0, request=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest configuration: a 128 x 64 run with a refined slab;
        # launches and their latency count
        _case("vortex2d", "D2Q9", "RR", (128, 64), 2, 16, slab=True, dtau=0.01, size=5.0),
        # a short request of the server: create, initialise, step, read, close
        _case("request2d_fp16", "D2Q9", "RR", (80, 80), 2, 100, storage="fp16", dtau=1e-3,
              ic="pulse", size=2.5, ma=0.15, request=True),
        # a medium 2D run of the server (three levels, one chunk of 25 steps)
        _case("serve2d_fp16", "D2Q9", "RR", (592, 592), 3, 25, storage="fp16", dtau=3e-4,
              ic="pulse", size=18.5),
        # the 2D benchmark: 33 runs of the 512^2 acoustic pulse, one launch
        # for all of them, in both storages
        _case("pulse2d_x33", "D2Q9", "RR", (512, 512), 2, 10, batch=33, ma=0.0, ic="pulse"),
        _case("pulse2d_x33_fp16", "D2Q9", "RR", (512, 512), 2, 10, batch=33, storage="fp16",
              ic="pulse"),
        # the same layout with the hybrid collision, the paper's remedy
        _case("hrr2d_x16", "D2Q9", "HRR", (512, 512), 2, 6, batch=16),
        # the headline: vortex column in 256^3 with a refined half (67 M nodes)
        _case("vortex3d", "D3Q19", "RR", (256, 256, 256), 2, 4, slab=True, dtau=5e-5, size=8.0),
        # a 3D slab in binary16 storage
        _case("slab3d_fp16", "D3Q19", "RR", (160, 160, 160), 2, 6, slab=True, storage="fp16",
              ic="pulse", size=5.0),
        # three nested levels on the largest velocity set
        _case("pulse3d", "D3Q27", "RR", (192, 192, 192), 3, 4, ma=0.0, ic="pulse", size=4.0),
        # a small 3D run of the server
        _case("serve3d_fp16", "D3Q19", "RR", (80, 80, 80), 2, 25, storage="fp16", dtau=1e-3,
              ic="pulse", size=2.5),
        # the hybrid collision in 3D
        _case("hrr3d", "D3Q19", "HRR", (96, 96, 96), 2, 6),
        # plain collision, one level, odd sides (ragged rows and tiles)
        _case("bgk3d_odd", "D3Q27", "BGK", (161, 97, 83), 1, 12, dtau=5e-3, ic="pulse", size=5.0),
    ]


def _layout(c):
    """Per level: node counts (x, y, z), the box in parent units, bounded axes."""
    D = 2 if c["lattice"] == "D2Q9" else 3
    n = [c["nx"], c["ny"], c["nz"]]
    out = [dict(n=tuple(n), lo=None, hi=None, boxed=(False,) * 3, origin=(0.0,) * 3, h=1.0)]
    per = [True] * 3
    for l in range(1, c["levels"]):
        lo, hi, boxed, m, org = [0] * 3, [1] * 3, [False] * 3, [1] * 3, [0.0] * 3
        for a in range(D):
            if l == 1 and c["slab"]:
                lo[a], hi[a] = (n[0] // 2, n[0]) if a == 0 else (0, n[a])
            else:
                lo[a] = n[a] // 4
                hi[a] = n[a] - lo[a] - (0 if per[a] else 1)
            whole = per[a] and lo[a] == 0 and hi[a] == n[a]
            boxed[a] = not whole
            m[a] = 2 * n[a] if whole else 2 * (hi[a] - lo[a]) + 1
            org[a] = out[-1]["origin"][a] + lo[a] * out[-1]["h"]
        per = [per[a] and not boxed[a] for a in range(3)]
        n = m
        out.append(dict(n=tuple(m), lo=tuple(lo), hi=tuple(hi), boxed=tuple(boxed),
                        origin=tuple(org), h=out[-1]["h"] / 2))
    return out


def _active(c):
    """Updated nodes per level (the parent nodes inside a child's ring are not)."""
    lay, out = _layout(c), []
    for l, v in enumerate(lay):
        k = v["n"][0] * v["n"][1] * v["n"][2]
        if l + 1 < len(lay):
            ch = lay[l + 1]
            k -= math.prod(ch["hi"][a] - ch["lo"][a] - 3 if ch["boxed"][a] else v["n"][a]
                           for a in range(3))
        out.append(k)
    return out


def work(case):
    """Every updated node's populations read and written once per step (the
    read-out: read once, and four binary32 values written)."""
    q, s = Q[case["lattice"]], 2 if case["storage"] == "fp16" else 4
    act = _active(case)
    upd = case["steps"] * case["batch"] * sum(2 ** l * k for l, k in enumerate(act))
    nodes = case["batch"] * sum(math.prod(v["n"]) for v in _layout(case))
    per_node = {"D2Q9": 200, "D3Q19": 500, "D3Q27": 800}[case["lattice"]]
    return {"bytes": upd * 2 * q * s + case["batch"] * sum(act) * q * s + nodes * 16,
            "flops": upd * per_node}


def draw(rng):
    while True:
        lattice = rng.choice(["D2Q9", "D2Q9", "D3Q19", "D3Q27"])
        collision = rng.choice(["RR", "RR", "RR", "REG", "BGK", "HRR"])
        logint = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
        if lattice == "D2Q9":
            dims = (logint(64, 1024), logint(64, 1024), 1)
            batch = rng.choice([1, 1, logint(2, 33)])
        else:
            dims = (logint(48, 160), logint(48, 160), logint(48, 160))
            batch = rng.choice([1, 1, 1, 2, 3])
        levels = rng.randint(1, 3)
        slab = levels == 2 and rng.random() < 0.4
        if slab:
            dims = (dims[0] + dims[0] % 2,) + dims[1:]
        storage = rng.choice(["fp32", "fp16"])
        ma = rng.uniform(0.05, 0.2)
        if storage == "fp32" and rng.random() < 0.3:
            ma = 0.0
        dtau = math.exp(rng.uniform(math.log(1e-3 if collision == "BGK" else 1e-5),
                                    math.log(1e-2)))
        side = min(dims[:2] if lattice == "D2Q9" else dims)
        c = _case("", lattice, collision, dims, levels, rng.randint(2, 25), storage=storage,
                  slab=slab, batch=batch, dtau=dtau, ma=ma,
                  # (binary16 storage is for the weak acoustic pulses: a strong
                  # vortex is resolved to a few binary16 digits only)
                  ic=rng.choice(["vortex", "pulse"]) if ma and storage == "fp32" else "pulse",
                  size=max(2.5, side / 28.0),
                  request=lattice == "D2Q9" and batch == 1 and side < 200 and rng.random() < 0.3)
        del c["name"]
        if work(c)["bytes"] <= 0.5 * max(work(x)["bytes"] for x in listed()):
            return c


def _ics(c, seed):
    """The initial state of every run of the batch, from the seed."""
    rng = random.Random(seed * 1000003 + 17)
    u0 = c["ma"] * CS
    out = []
    for _ in range(c["batch"]):
        # across the refined boxes' upstream faces, so that every level and
        # every interface has something to do
        x = 0.5 if c["slab"] or c["levels"] == 1 else (0.27 if c["levels"] == 2 else 0.34)
        at = [c["nx"] * x, c["ny"] * 0.5, c["nz"] * 0.5]
        at = [p + rng.uniform(-0.03, 0.03) * n for p, n in zip(at, (c["nx"], c["ny"], c["nz"]))]
        if c["lattice"] == "D2Q9":
            at[2] = 0.0
        k = rng.uniform(0.8, 1.2)
        out.append(dict(kind=c["ic"], u0=(u0, 0.0, 0.0), center=tuple(at), radius=c["size"] * k,
                        amplitude=1e-3 * k, eps=0.05 * CS * k))
    return out


def _open(c, ics):
    lay = _layout(c)
    dims = (c["nx"], c["ny"], c["nz"])
    h = mlbm.Lbm(c["lattice"], c["collision"], 0.5 + c["dtau"], dims,
                 [(v["lo"], v["hi"]) for v in lay[1:]], storage=c["storage"], batch=c["batch"],
                 u_ref=(c["ma"] * CS, 0.0, 0.0), sigma=SIGMA, torch_allocator=True,
                 stream=torch.cuda.current_stream().cuda_stream)
    for b, ic in enumerate(ics):
        h.init_analytic(ic, b)
    return h


def prepare(case, seed):
    ics = _ics(case, seed)
    nodes = [math.prod(v["n"]) for v in _layout(case)]
    B = case["batch"]
    out = [dict(rho=torch.zeros(B, n, device="cuda"), u=torch.zeros(B, 3, n, device="cuda"))
           for n in nodes]
    return dict(case=case, ics=ics, out=out, run=None if case["request"] else _open(case, ics))


def run(state):
    c = state["case"]
    h = state["run"] if state["run"] is not None else _open(c, state["ics"])
    h.step(c["steps"])
    for l, out in enumerate(state["out"]):
        for b in range(c["batch"]):
            h.macros_device(l, out["rho"][b].data_ptr(), out["u"][b].data_ptr(), run=b)
    if state["run"] is None:
        h.close()
    return state["out"]


# --------------------------------------------------------------------------
# The same pass in 64 bits with plain torch: dense arrays [q, run, z, y, x],
# two arrays per level, the paper's order of operations.
# --------------------------------------------------------------------------

PAIRS = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
THIRD = ((0, 0, 1), (0, 0, 2), (1, 1, 0), (1, 1, 2), (2, 2, 0), (2, 2, 1), (0, 1, 2))


class _Lattice:
    def __init__(self, name, dev):
        D = 2 if name == "D2Q9" else 3
        self.D = D
        xi = [(x, y, z) for z in (range(-1, 2) if D == 3 else (0,)) for y in range(-1, 2)
              for x in range(-1, 2)]
        if name == "D3Q19":
            xi = [c for c in xi if sum(map(abs, c)) < 3]
        w = {"D2Q9": (4 / 9, 1 / 9, 1 / 36), "D3Q19": (1 / 3, 1 / 18, 1 / 36),
             "D3Q27": (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[name]
        self.xi, self.q = xi, len(xi)
        H3 = lambda c, a, b: c[a] * c[a] * c[b] - c[b] / 3.0  # noqa: E731
        rows = []  # coefficients of (a0, a1[3], a2[6], a3[7]) in the expansion, eq. fEqH
        for c in xi:
            r = [1.0] + [3.0 * c[a] for a in range(3)]
            r += [4.5 * (c[a] * c[b] - (a == b) / 3.0) * (1 if a == b else 2) for a, b in PAIRS]
            t = [0.0] * 7
            if name == "D3Q19":
                for b in range(3):
                    a, d = [k for k in range(3) if k != b]
                    hp, hm = H3(c, a, b) + H3(c, d, b), H3(c, a, b) - H3(c, d, b)
                    t[THIRD.index((a, a, b))] += 13.5 * hp + 4.5 * hm
                    t[THIRD.index((d, d, b))] += 13.5 * hp - 4.5 * hm
            else:
                for k, (a, b, d) in enumerate(THIRD):
                    if D == 2 and 2 in (a, b, d):
                        continue
                    t[k] = 13.5 * H3(c, a, d) if a == b else 27.0 * c[0] * c[1] * c[2]
            if D == 2:
                r[6] = r[8] = r[9] = 0.0
            rows.append([w[sum(map(abs, c))] * v for v in r + t])
        T = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
        self.C = T(rows)
        self.E = T([[1.0] * self.q] + [[float(c[a]) for c in xi] for a in range(3)])
        self.H2 = T([[c[a] * c[b] - (a == b) / 3.0 for c in xi] for a, b in PAIRS])

    def moments(self, f):
        m = self.E @ f
        return m[0], m[1:] / m[0]

    def equilibrium_moments(self, rho, u):
        rows = [rho] + [rho * u[a] for a in range(3)]
        rows += [rho * u[a] * u[b] for a, b in PAIRS]
        rows += [rho * u[a] * u[b] * u[c] for a, b, c in THIRD]
        return torch.stack(rows)

    def split(self, f):
        """rho, u and the off-equilibrium part of f [q, N]."""
        rho, u = self.moments(f)
        return rho, u, f - self.C @ self.equilibrium_moments(rho, u)

    def collide(self, f, coll, tau, S=None):
        rho, u = self.moments(f)
        M = self.equilibrium_moments(rho, u)
        feq = self.C @ M
        om = 1.0 - 1.0 / tau
        if coll == "BGK":
            return feq + om * (f - feq)
        a1 = self.H2 @ (f - feq)
        if self.D == 2:
            a1[2] = a1[4] = a1[5] = 0.0
        if coll == "HRR":
            a1 = SIGMA * a1 - (1.0 - SIGMA) * 2.0 * tau / 3.0 * rho * S
        at = lambda a, b: a1[PAIRS.index((min(a, b), max(a, b)))]  # noqa: E731
        M1 = torch.zeros_like(M)
        M1[4:10] = a1
        if coll != "REG":
            for k, (a, b, c) in enumerate(THIRD):
                M1[10 + k] = u[a] * at(b, c) + u[b] * at(a, c) + u[c] * at(a, b)
        return feq + om * (self.C @ M1)


class _Exact:
    CHUNK = 1 << 23

    def __init__(self, c, seed, dev):
        self.c, self.dev = c, dev
        self.L = _Lattice(c["lattice"], dev)
        self.D, self.B = self.L.D, c["batch"]
        self.lev = _layout(c)
        ics = _ics(c, seed)
        tau, per = 0.5 + c["dtau"], [True] * 3
        for l, v in enumerate(self.lev):
            per = [per[a] and not v["boxed"][a] for a in range(3)]
            v.update(tau=tau, per=list(per), nsteps=0)
            tau = 2.0 * tau - 0.5
            rho, u = zip(*(self._fields(v, ic) for ic in ics))
            rho, u = torch.stack(rho), torch.stack(u, 1)
            shape = rho.shape
            v["shape"] = shape
            f = self.L.C @ self.L.equilibrium_moments(rho.flatten(), u.reshape(3, -1))
            v["post"] = f.reshape(-1, *shape)
            v["vel"] = u
            if l:
                p = self.lev[l - 1]
                seen = self._window(l, p["rho0"]), self._window(l, p["u0"])
                first = [torch.cat([r[None], w, torch.zeros(self.L.q, *r.shape, device=dev,
                                                            dtype=torch.float64)])
                         for r, w in zip(*seen)]
                v["hist"] = [first, first, first]
                if c["collision"] == "HRR":
                    s = self._window(l, self._strain(p["u0"]))
                    v["shist"] = [s, s, s]
            v["rho0"], v["u0"] = rho, u
        for v in self.lev:
            del v["rho0"], v["u0"]

    def _fields(self, v, ic):
        dom, ax = (self.c["nx"], self.c["ny"], self.c["nz"]), []
        for a in range(3):
            x = v["origin"][a] + v["h"] * torch.arange(v["n"][a], dtype=torch.float64,
                                                       device=self.dev)
            d = torch.remainder(x, dom[a]) - ic["center"][a]
            ax.append(d - dom[a] * torch.round(d / dom[a]))
        dx, dy, dz = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
        zero = torch.zeros(v["n"][2], v["n"][1], v["n"][0], dtype=torch.float64, device=self.dev)
        R = ic["radius"]
        u = [zero + ic["u0"][0], zero.clone(), zero.clone()]
        if ic["kind"] == "vortex":
            g = torch.exp(-(dx * dx + dy * dy) / (2.0 * R * R)) + zero
            rho = 1.0 - 1.5 * ic["eps"] ** 2 * g * g
            u[0] = u[0] - ic["eps"] * (dy / R) * g
            u[1] = u[1] + ic["eps"] * (dx / R) * g
        else:
            r2 = dx * dx + dy * dy + (dz * dz if self.D == 3 else 0.0)
            rho = 1.0 + ic["amplitude"] * torch.exp(-r2 / (2.0 * R * R)) + zero
        return rho, torch.stack(u)

    def _chunks(self, fn, *arrays):
        """fn over the nodes of arrays [k, ...], a piece at a time."""
        n = arrays[0][0].numel()
        flat = [a.reshape(a.shape[0], -1) for a in arrays]
        parts = [fn(*(a[:, i:i + self.CHUNK].contiguous() for a in flat))
                 for i in range(0, n, self.CHUNK)]
        return torch.cat(parts, 1).reshape(-1, *arrays[0].shape[1:])

    # dims of a field [k, run, z, y, x]: axis a is dim 4 - a
    def _stream(self, f):
        out = torch.empty_like(f)
        for i, c in enumerate(self.L.xi):
            out[i] = torch.roll(f[i], (c[2], c[1], c[0]), (1, 2, 3))
        return out

    def _strain(self, u):
        g = [[0.5 * (torch.roll(u[b], -1, 3 - a) - torch.roll(u[b], 1, 3 - a)) for b in range(3)]
             for a in range(3)]
        return torch.stack([0.5 * (g[a][b] + g[b][a]) for a, b in PAIRS])

    def _faces(self, l):
        v = self.lev[l]
        return [(a, s) for a in range(self.D) if v["boxed"][a] for s in (0, 1)]

    def _window(self, l, field):
        """The parent's field on every face plane of level l's box, one cell
        past its edges on bounded axes."""
        v, p = self.lev[l], self.lev[l - 1]
        out = []
        squeeze = field.dim() == 4  # a scalar [run, z, y, x]
        field = field[None] if squeeze else field
        for a, s in self._faces(l):
            w = field
            for b in range(3):
                if b >= self.D:
                    continue
                if b == a:
                    at = [v["hi"][a] if s else v["lo"][a]]
                elif v["boxed"][b]:
                    at = range(v["lo"][b] - 1, v["hi"][b] + 2)
                else:
                    continue
                at = torch.tensor([k % p["n"][b] for k in at], device=self.dev)
                w = w.index_select(4 - b, at)
            out.append(w[0] if squeeze else w)
        return out

    def _to_child(self, l, a, w):
        """Cubic interpolation along the tangent axes of face axis a (eq. spaceInt)."""
        v = self.lev[l]
        for b in range(self.D):
            if b == a:
                continue
            d = 4 - b
            if v["boxed"][b]:
                m = w.shape[d] - 2
                cut = lambda k, n: w.narrow(d, k, n)  # noqa: E731
                even = cut(1, m)
                odd = (9.0 * (cut(1, m - 1) + cut(2, m - 1)) - cut(0, m - 1) - cut(3, m - 1)) / 16.0
                out = torch.empty(*w.shape[:d], 2 * m - 1, *w.shape[d + 1:], dtype=w.dtype,
                                  device=w.device)
                ix = torch.arange(2 * m - 1, device=w.device)
            else:
                m = w.shape[d]
                even = w
                odd = (9.0 * (w + torch.roll(w, -1, d)) - torch.roll(w, 1, d)
                       - torch.roll(w, -2, d)) / 16.0
                out = torch.empty(*w.shape[:d], 2 * m, *w.shape[d + 1:], dtype=w.dtype,
                                  device=w.device)
                ix = torch.arange(2 * m, device=w.device)
            out.index_copy_(d, ix[0::2], even)
            out.index_copy_(d, ix[1::2], odd)
            w = out
        return w

    def _boundary(self, l, hist, wt):
        """(face axis, index on it, the history interpolated to its child nodes)."""
        v = self.lev[l]
        for k, (a, s) in enumerate(self._faces(l)):
            g = sum(t * h[k] for t, h in zip(wt, hist) if t != 0.0)
            yield a, (v["n"][a] - 1 if s else 0), self._to_child(l, a, g)

    def _at(self, a, i):
        ix = [slice(None)] * 5
        ix[4 - a] = slice(i, i + 1)
        return tuple(ix)

    def _tn(self, l):
        """Boxes of the TN ring: slices on level l and, with `pad` neighbours, on its child."""
        v, c = self.lev[l], self.lev[l + 1]
        for a in range(self.D):
            if not c["boxed"][a]:
                continue
            for s in (0, 1):
                par, ch = [], []
                for b in range(3):
                    E = c["hi"][b] - c["lo"][b]
                    if b >= self.D or not c["boxed"][b]:
                        r = range(v["n"][b])
                        par.append(torch.tensor(list(r), device=self.dev))
                        ch.append([2 * k if b < self.D else 0 for k in r])
                        continue
                    r = [E - 1 if s else 1] if b == a else list(range(1, E))
                    par.append(torch.tensor([(c["lo"][b] + k) % v["n"][b] for k in r],
                                            device=self.dev))
                    ch.append([2 * k for k in r])
                yield par, ch

    def _take(self, f, ix):
        for b in range(3):
            f = f.index_select(4 - b, ix[b])
        return f

    def _put(self, f, ix, val):
        Z, Y, X = torch.meshgrid(ix[2], ix[1], ix[0], indexing="ij")
        f[:, :, Z, Y, X] = val

    def _child_at(self, l, ch, off):
        c = self.lev[l + 1]
        return [torch.tensor([(k + off[b]) % c["n"][b] for k in ch[b]], device=self.dev)
                for b in range(3)]

    def _restrict(self, l):
        v, c, L = self.lev[l], self.lev[l + 1], self.L
        resc = 2.0 * v["tau"] / c["tau"]
        offs = [(x, y, z) for x in (-1, 0, 1) for y in (-1, 0, 1)
                for z in ((-1, 0, 1) if self.D == 3 else (0,))]
        for par, ch in self._tn(l):
            f1s = 0.0
            for o in offs:
                w = math.prod(0.5 if o[b] == 0 else 0.25 for b in range(self.D))
                f = self._take(c["pre"], self._child_at(l, ch, o))
                rho, u, f1 = L.split(f.reshape(L.q, -1))
                f1s = f1s + w * f1
                if not any(o):
                    eq = L.C @ L.equilibrium_moments(rho, u)
                    shape, vel = f.shape, u
            self._put(v["pre"], par, (eq + resc * f1s).reshape(shape))
            if self.c["collision"] == "HRR":
                self._put(v["vel"], par, vel.reshape(3, *shape[1:]))
                S = self._take(c["sused"], self._child_at(l, ch, (0, 0, 0)))
                v["given"].append((par, 2.0 * S))

    def _parent_strain(self, l):
        """The strain rate of level l on its child's box surface at t+1."""
        v, c, L = self.lev[l], self.lev[l + 1], self.L
        for par, ch in self._tn(l):
            f = torch.stack([self._take(c["post"][i:i + 1],
                                        self._child_at(l, ch, tuple(-k for k in xi)))[0]
                             for i, xi in enumerate(L.xi)])
            _, u = L.moments(f.reshape(L.q, -1))
            self._put(v["vel"], par, u.reshape(3, *f.shape[1:]))
        c["shist"] = c["shist"][1:] + [self._window(l + 1, self._strain(v["vel"]))]

    def advance(self, l, wt, first=False):
        v, L, hrr = self.lev[l], self.L, self.c["collision"] == "HRR"
        v["pre"] = self._stream(v["post"])
        v["given"] = []
        if l:
            resc = v["tau"] / (2.0 * self.lev[l - 1]["tau"])
            for a, i, g in self._boundary(l, v["hist"], wt):
                flat = g.reshape(g.shape[0], -1)
                f = L.C @ L.equilibrium_moments(flat[0], flat[1:4]) + resc * flat[4:]
                v["pre"][self._at(a, i)] = f.reshape(-1, *g.shape[1:])
        if hrr:
            v["vel"] = self._chunks(lambda f: L.moments(f)[1], v["pre"])
        if l + 1 < len(self.lev):
            c = self.lev[l + 1]
            new = []
            for w in self._window(l + 1, v["pre"]):
                rho, u, f1 = L.split(w.reshape(L.q, -1))
                new.append(torch.cat([rho[None], u, f1]).reshape(-1, *w.shape[1:]))
            c["hist"] = c["hist"][1:] + [new]
            wa = (0.0, 0.5, 0.5) if v["nsteps"] == 0 else (-0.125, 0.75, 0.375)
            self.advance(l + 1, wa, True)
            self.advance(l + 1, (0.0, 0.0, 1.0))
            self._restrict(l)
        S = None
        if hrr:
            S = self._strain(v["vel"])
            for par, s in v["given"]:
                self._put(S, par, s)
        coll, tau = self.c["collision"], v["tau"]
        if hrr:
            v["post"] = self._chunks(lambda f, s: L.collide(f, coll, tau, s), v["pre"], S)
            if l:
                if first:
                    self._parent_strain(l - 1)
                for a, i, g in self._boundary(l, v["shist"], wt):
                    at = self._at(a, i)
                    f = v["pre"][at]
                    S[at] = 0.5 * g
                    out = L.collide(f.reshape(L.q, -1), coll, tau, 0.5 * g.reshape(6, -1))
                    v["post"][at] = out.reshape(f.shape)
            v["sused"] = S
        else:
            v["post"] = self._chunks(lambda f: L.collide(f, coll, tau), v["pre"])
        v["nsteps"] += 1

    def outputs(self):
        res = []
        for l, v in enumerate(self.lev):
            m = self._chunks(lambda f: torch.cat([(r := self.L.moments(f))[0][None], r[1]]),
                             v["post"])
            if self.D == 2:
                m[3] = 0.0
            if l + 1 < len(self.lev):
                c, ix = self.lev[l + 1], []
                for b in range(3):
                    lo, hi = (c["lo"][b] + 2, c["hi"][b] - 2) if c["boxed"][b] else \
                        (0, v["n"][b] - 1)
                    ix.append(slice(lo, hi + 1))
                m[:, :, ix[2], ix[1], ix[0]] = float("nan")
            m = m.reshape(4, self.B, -1)
            res.append(dict(rho=m[0], u=m[1:].transpose(0, 1).contiguous()))
        return res


def exact(case, seed, device="cuda"):
    x = _Exact(case, seed, device)
    for _ in range(case["steps"]):
        x.advance(0, None)
    return x.outputs()
