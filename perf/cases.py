"""Performance cases of the adaptive ray trace: calls that users of the library make, with the
sizes of the configurations in ``bench.py`` and the tests (and odd-sized relatives of them).

Families (key ``family`` of a case):

* ``trace``    -- one forward trace of all sources (``Grid.trace``);
* ``backward`` -- one reverse sweep (``Grid.trace_backward``);
* ``autograd`` -- forward and backward through ``ARTFunction``, as a fit of the density does;
* ``substep``  -- one ionization substep: trace, ``dt_substep``, ``xn_update``;
* ``xn``       -- ``xn_update`` alone (it runs once per step on every cell of a large grid).

``exact`` restates the method (Sec. 2.1 and 2.3 of Kim, Kim, Ostriker & Skinner 2017) in FP64
torch arithmetic: breadth-first over the HEALPix levels, all rays of a level side by side.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1711_06277_gb300 import art

_TRACE = dict(family="trace", field="lognormal", sigma_ln=1.5, density=1.0, placement="random",
              sigma_H=10.0, sigma_d=0.0, bins=1, force=True, energy=False, rotate=False,
              d_max=0.0, level0=4, m_ray=4.0, tau_max=30.0)


def _trace_case(name, shape, nsrc, **kw):
    nx, ny, nz = shape
    c = dict(_TRACE, name=name, nx=nx, ny=ny, nz=nz, nsrc=nsrc)
    c.update(kw)
    return c


def listed():
    return [
        # one source in a small uniform box: the latency of a single call (a code's unit test,
        # a sub-grid around one star)
        _trace_case("trace_32_1src", (32, 32, 32), 1, field="uniform", sigma_H=5.0,
                    placement="centre"),
        # one star in a turbulent cloud
        _trace_case("trace_128_1src", (128, 128, 128), 1, placement="cell"),
        # a cluster in a turbulent cloud
        _trace_case("trace_256_64src", (256, 256, 256), 64, sigma_ln=2.0),
        # part of the largest workload (512^3, 1024 sources): its grid and ionized gas, with as
        # many sources as one rank of a split run holds
        _trace_case("trace_512_64src", (512, 512, 512), 64, sigma_ln=2.0, density=0.1, sigma_H=0.1),
        # weak-scaling set-up (Sec. 3.1): a source at the centre of every 32^3 block, rays cut
        # at 0.6 of a block
        _trace_case("trace_128_blocks_dmax", (128, 128, 128), 64, field="uniform", sigma_H=2.0,
                    placement="blocks", d_max=0.6 * 32 / 128),
        # radiation pressure on dust with two frequency bins and a per-step rotation, in a box
        # without round numbers, at the paper's default depth limit
        _trace_case("trace_odd_dust_2bin", (97, 130, 61), 5, sigma_H=20.0, sigma_d=6.0, bins=2,
                    density=0.3, energy=True, rotate=True, level0=3, tau_max=7.0),
        # gradient of a loss on the photoionization rate
        _trace_case("backward_128_16src", (128, 128, 128), 16, family="backward"),
        # gradient of a loss on rate and force, with dust, in an odd box
        _trace_case("backward_odd_force_dust", (75, 66, 90), 6, family="backward", sigma_H=6.0,
                    sigma_d=1.5, level0=3),
        # one iteration of a fit of the density and the luminosities
        _trace_case("autograd_64_8src", (64, 64, 64), 8, family="autograd", force=False),
        # one substep of an expanding ionization front (Sec. 3.3.1): sharp front, dark outside
        _trace_case("substep_128_front", (128, 128, 128), 1, family="substep", field="bubble",
                    placement="cell", sigma_H=109.0 * 128, force=False),
        # neutral-fraction update of the largest grid (Eq. e:xn3)
        dict(name="xn_512_b", family="xn", ncell=512 ** 3, method="b"),
        # the exact quadratic update (Eq. e:xn2)
        dict(name="xn_256_a", family="xn", ncell=256 ** 3, method="a"),
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    family = rng.choice(["trace"] * 4 + ["backward"] * 2 + ["autograd", "substep", "xn"])
    if family == "xn":
        return dict(family="xn", ncell=logint(1000, 512 ** 3), method=rng.choice(["a", "b"]))
    side = logint(24, {"trace": 400, "backward": 200, "autograd": 128, "substep": 256}[family])
    shape = [max(8, int(side * rng.uniform(0.6, 1.0))) for _ in range(3)]
    cells = shape[0] * shape[1] * shape[2]
    # at most a quarter of the largest listed case's rays through cells (a reverse sweep walks
    # every ray twice and gathers more)
    room = 16 * 512 ** 3 / (1 if family == "trace" else 8)
    m_ray = rng.choice([4.0, 4.0, 4.0, 2.0, 8.0, 16.0])
    nsrc = min(logint(1, 64), max(1, int(room / (cells * m_ray / 4.0))))
    c = _trace_case("", shape, nsrc, family=family, sigma_ln=rng.choice([1.5, 2.0]),
                    sigma_H=math.exp(rng.uniform(math.log(1.0), math.log(20.0))),
                    level0=rng.choice([2, 3, 4, 4, 5]), m_ray=m_ray,
                    tau_max=rng.choice([7.0, 30.0]), rotate=rng.random() < 0.3)
    del c["name"]
    if family in ("trace", "backward") and rng.random() < 0.4:
        c["sigma_d"] = rng.uniform(0.5, 6.0)
    if family == "trace":
        c["bins"] = 2 if c["sigma_d"] > 0 and rng.random() < 0.5 else 1
        c["force"] = rng.random() < 0.7
        c["energy"] = rng.random() < 0.3
    if family in ("trace", "backward") and rng.random() < 0.2:
        c["d_max"] = rng.uniform(0.1, 0.5)
    if family == "backward":
        c["force"] = rng.random() < 0.5
    if family == "autograd":
        c["force"] = False
    if family == "substep":
        c.update(field="bubble", nsrc=1, placement="cell", sigma_H=109.0 * 128, force=False)
    return c


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    return g


def _lognormal(shape, sigma_ln, gen):
    """Lognormal density of mean 1 with a k^-4 power spectrum, shape (nz, ny, nx), float32."""
    dev = _device()
    nz, ny, nx = shape
    side = max(shape)
    wk = torch.fft.rfftn(torch.randn(shape, generator=gen, device=dev))
    kz, ky = (torch.fft.fftfreq(n, 1.0 / side, device=dev) for n in (nz, ny))
    kx = torch.fft.rfftfreq(nx, 1.0 / side, device=dev)
    k2 = kz[:, None, None] ** 2 + ky[:, None] ** 2 + kx ** 2
    k2[0, 0, 0] = math.inf
    f = torch.fft.irfftn(wk / k2, s=shape)
    f = f / f.std()
    rho = torch.exp(sigma_ln * f - 0.5 * sigma_ln ** 2)
    return (rho / rho.mean()).contiguous()


def _sources(case, rng):
    """Positions (nsrc, 3) in the box [0, n dx)^3 and luminosities summing to 1."""
    n = np.array([case["nx"], case["ny"], case["nz"]], dtype=np.float64)
    dx = 1.0 / n.max()
    k = case["nsrc"]
    if case["placement"] == "centre":
        pos = (0.5 * n * dx)[None, :]
    elif case["placement"] == "cell":
        pos = ((np.floor(n * rng.uniform(0.35, 0.65, 3)) + 0.5) * dx)[None, :]
    elif case["placement"] == "blocks":
        b = [(np.arange(int(m) // 32) + 0.5) * 32 * dx for m in n]
        pos = np.stack(np.meshgrid(*b, indexing="ij"), -1).reshape(-1, 3)
        return pos, np.full(len(pos), 1.0 / len(pos))
    else:
        pos = rng.uniform(1e-3, 1.0 - 1e-3, (k, 3)) * n * dx
    lum = 1.0 / (1e3 - rng.random(k) * (1e3 - 1.0))  # dN/dL ~ L^-2 on [1e-3, 1]
    return pos, lum / lum.sum()


def _rotation(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


def _inputs(case, seed):
    """Fields, sources, loss weights and trace parameters of a case (device tensors, numpy)."""
    gen, rng = _generator(seed), np.random.default_rng(seed)
    dev = _device()
    if case["family"] == "xn":
        n = case["ncell"]
        u = torch.rand((3, n), generator=gen, device=dev)
        x = 10.0 ** (-4.0 * u[0])                       # from ionized to neutral gas
        gamma = 10.0 ** (6.0 * u[1] - 3.0)
        gamma[u[1] < 0.1] = 0.0                         # shielded cells
        return dict(xn=x, gamma=gamma, nH=100.0 * 10.0 ** (2.0 * u[2] - 1.0), alpha=2e-4, dt=5.0)
    shape = (case["nz"], case["ny"], case["nx"])
    d = dict(shape=shape, dx=1.0 / max(shape))
    d["pos"], d["L"] = _sources(case, rng)
    if case["field"] == "uniform":
        rho = torch.full(shape, 1.0, device=dev)
    elif case["field"] == "bubble":                     # x_n around the first source
        z, y, x = (torch.arange(m, device=dev, dtype=torch.float32) + 0.5 for m in shape)
        c = d["pos"][0] / d["dx"]
        r = torch.sqrt((z[:, None, None] - c[2]) ** 2 + (y[:, None] - c[1]) ** 2 + (x - c[0]) ** 2)
        front = max(shape) * rng.uniform(0.25, 0.3)
        rho = 1e-4 + (1.0 - 1e-4) * torch.sigmoid((r - front) / 1.5)
    else:
        rho = _lognormal(shape, case["sigma_ln"], gen)
    d["nH0"] = (case["density"] * rho).contiguous()
    d["nH"] = rho if case["sigma_d"] > 0 else None
    d["Ln"] = 3.0 * d["L"][::-1].copy() if case["bins"] == 2 else None
    d["w"] = torch.rand(shape, generator=gen, device=dev)
    d["v"] = 2.0 * torch.rand((3,) + shape, generator=gen, device=dev) - 1.0 \
        if case["family"] == "backward" and case["force"] else None
    d["rot"] = _rotation(rng) if case["rotate"] else None
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    if case["family"] == "xn":
        d["nH0"] = torch.empty_like(d["xn"])
        return dict(d, case=case)
    if case["family"] == "substep":
        d["xn"] = d["nH0"].clone()
        d["nH"] = torch.ones_like(d["xn"])
        d["nH0_out"] = torch.empty_like(d["xn"])
    if case["family"] == "autograd":
        d["log_nH0"] = torch.log(d["nH0"])
        d["L"] = torch.from_numpy(d["L"])
    grid = art.Grid(d["nH0"], d["dx"], nH=d["nH"] if case["sigma_d"] > 0 else None)
    if case["family"] != "autograd":
        grid.add_sources(d["pos"], d["L"])
        if d["Ln"] is not None:
            grid.set_nonionizing(d["Ln"])
    params = art.Params(level0=case["level0"], m_ray=case["m_ray"], tau_max=case["tau_max"],
                        sigma_H=case["sigma_H"], sigma_d=case["sigma_d"], rot=d["rot"],
                        d_max=case["d_max"])
    return dict(d, case=case, grid=grid, params=params)


def run(state):
    s, case = state, state["case"]
    family = case["family"]
    if family == "xn":
        x = s["xn"].clone()  # the call updates in place
        art.xn_update(s["gamma"], s["nH"], x, s["alpha"], s["dt"], nH0_out=s["nH0"],
                      method=case["method"])
        return {"xn": x, "nH0": s["nH0"]}
    if family == "trace":
        o = s["grid"].trace(s["params"], force=case["force"], energy=case["energy"], stats=False)
        return {k: o[k] for k in ("gamma", "force", "energy") if o[k] is not None}
    if family == "backward":
        grad, dL, _ = s["grid"].trace_backward(s["params"], s["w"], stats=False, v=s["v"])
        return {"grad": grad, "dL": dL}
    if family == "autograd":
        q = s["log_nH0"].detach().requires_grad_()
        L = s["L"].detach().requires_grad_()
        gamma = art.ARTFunction.apply(q, L, s["grid"], s["params"], s["pos"])
        (gamma * s["w"]).sum().backward()
        return {"gamma": gamma.detach(), "grad": q.grad, "dL": L.grad}
    gamma = s["grid"].trace(s["params"], force=False, stats=False)["gamma"]
    dt = art.dt_substep(gamma, s["nH"], s["xn"], 1.0, 0.1)
    x = s["xn"].clone()
    art.xn_update(gamma, s["nH"], x, 1.0, float(dt.cpu()), nH0_out=s["nH0_out"])
    return {"gamma": gamma, "dt": dt, "xn": x, "nH0": s["nH0_out"]}


def _crossings(case):
    """Estimate of a trace's crossings in a thin medium: 12 4^l0 rays per source out to
    r_max(l0), beyond it about 3 m_ray per cell (the splitting keeps m_ray to 4 m_ray)."""
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["d_max"] > 0:
        cells = min(cells, 4.0 / 3.0 * math.pi * (case["d_max"] * max(case["nx"], case["ny"], case["nz"])) ** 3)
    if case["field"] == "bubble":
        cells *= 0.1                                     # rays end at the front
    reach = (3.0 * cells / (4.0 * math.pi)) ** (1.0 / 3.0)
    r0 = math.sqrt(3.0 / (math.pi * case["m_ray"])) * 2 ** case["level0"]
    base = 1.5 * 12 * 4 ** case["level0"] * min(r0, reach)
    beyond = 3.0 * case["m_ray"] * max(0.0, cells - 4.0 / 3.0 * math.pi * r0 ** 3)
    return case["nsrc"] * (base + beyond)


def work(case):
    """Per cell: fields in, outputs out. Per crossing of a trace: next face and segment (2),
    optical depth (2), attenuation (about 12), the four deposits (7); a reverse sweep walks
    twice and adds the derivative."""
    if case["family"] == "xn":
        return {"bytes": 20 * case["ncell"], "flops": (20 if case["method"] == "b" else 60) * case["ncell"]}
    cells = case["nx"] * case["ny"] * case["nz"]
    fields = 4 * (1 + (case["sigma_d"] > 0))
    fwd = fields + 4 * (1 + 3 * case["force"] + case["energy"])
    bwd = fields + 4 * (2 + 3 * case["force"])
    per_cell = {"trace": fwd, "backward": bwd, "autograd": fwd + bwd, "substep": fwd + 16}[case["family"]]
    per_cross = {"trace": 23 + 12 * (case["bins"] - 1), "backward": 60, "autograd": 83, "substep": 20}[case["family"]]
    return {"bytes": per_cell * cells, "flops": per_cross * _crossings(case)}


# ---------------------------------------------------------------------------------------
# the method in FP64
# ---------------------------------------------------------------------------------------
def _directions(level, pix, rot):
    """HEALPix nested pixel centres (Gorski et al. 2005), shape (k, 3); components below
    2^-24 count as zero."""
    ns = 1 << level
    face, q = pix // (ns * ns), pix % (ns * ns)
    x = torch.zeros_like(q)
    y = torch.zeros_like(q)
    for b in range(level):
        x |= ((q >> (2 * b)) & 1) << b
        y |= ((q >> (2 * b + 1)) & 1) << b
    row = face // 4
    ring = (row + 2) * ns - x - y - 1
    north, south = ring < ns, ring > 3 * ns
    cap = north | south
    nr = torch.where(north, ring, torch.where(south, 4 * ns - ring, torch.full_like(ring, ns)))
    shift = torch.where(cap, torch.zeros_like(ring), (ring - ns) % 2)
    a = nr.double() ** 2 / (3.0 * ns * ns)
    z = torch.where(cap, torch.where(north, 1.0 - a, a - 1.0), (4 * ns - 2 * ring).double() / (3.0 * ns))
    st = torch.where(cap, torch.sqrt(a * (2.0 - a)), torch.sqrt((1.0 - z) * (1.0 + z)))
    col = 2 * (face % 4) + (row != 1).long()
    jp = torch.div(col * nr + x - y + 1 + shift, 2, rounding_mode="floor")
    phi = math.pi * (2 * jp - shift - 1).double() / (4.0 * nr.double())
    v = torch.stack([st * torch.cos(phi), st * torch.sin(phi), z], -1)
    if rot is not None:
        v = v @ torch.as_tensor(rot, dtype=torch.float64, device=v.device).T
    return torch.where(v.abs() < 2.0 ** -24, torch.zeros_like(v), v)


def _phi(x):
    return torch.where(x > 0, -torch.expm1(-x) / torch.where(x > 0, x, torch.ones_like(x)), torch.ones_like(x))


def _dphi(x, phi):
    s = -1 / 2 + x * (1 / 3 + x * (-1 / 8 + x * (1 / 30 + x * (-1 / 144 + x / 840))))
    return torch.where(x < 1e-2, s, (torch.exp(-x) - phi) / torch.where(x < 1e-2, torch.ones_like(x), x))


class _Trace64:
    """The trace of one case in FP64, with its gradient."""

    def __init__(self, case, d):
        dev = _device()
        self.case, self.dev = case, dev
        nz, ny, nx = d["shape"]
        self.n = torch.tensor([nx, ny, nz], device=dev)
        self.stride = torch.tensor([1, nx, nx * ny], device=dev)
        self.dx = d["dx"]
        self.dV = self.dx ** 3
        h = d["nH0"].double().reshape(-1) * (case["sigma_H"] * self.dx)
        dust = 0.0 if d["nH"] is None else d["nH"].double().reshape(-1) * (case["sigma_d"] * self.dx)
        self.chiH, self.chi = h, h + dust
        self.chin = dust if case["bins"] == 2 else None
        self.u = torch.from_numpy(np.asarray(d["pos"]) / self.dx).to(dev)
        self.L = torch.as_tensor(np.asarray(d["L"]), dtype=torch.float64, device=dev)
        self.Ln = None if d["Ln"] is None else torch.from_numpy(d["Ln"]).to(dev)
        self.rot = d["rot"]
        unit = math.sqrt(3.0 / (math.pi * case["m_ray"]))
        self.rmax = [unit * 2.0 ** l for l in range(15)]
        far = torch.maximum(self.u, self.n - self.u).norm(dim=1)
        self.lmax = torch.full((len(self.L),), case["level0"], device=dev)
        for l in range(case["level0"], 13):
            self.lmax = torch.where((self.lmax == l) & (self.rmax[l] < far), l + 1, self.lmax)
        cells = nx * ny * nz
        self.G = torch.zeros(cells, dtype=torch.float64, device=dev)
        self.F = torch.zeros((3, cells), dtype=torch.float64, device=dev) if case["force"] else None

    def walk(self, l, src, pix, L, tau, Ln, taun, segment):
        """Walks rays of level l from entry to end; ``segment(rows, cell, n, ds, x, L, phi, xn,
        Ln)`` sees every segment. Returns what the rays carry at the end and which split."""
        case = self.case
        r0 = 0.0 if l == case["level0"] else self.rmax[l - 1]
        cut = case["d_max"] / self.dx if case["d_max"] > 0 else math.inf
        n = _directions(l, pix, self.rot)
        u = self.u[src]
        rend = torch.full_like(u[:, 0], math.inf).masked_fill(self.lmax[src] > l, self.rmax[l]).clamp(max=cut)
        p = u + r0 * n
        cell = torch.floor(p)
        cell = torch.where((p == cell) & (n < 0), cell - 1, cell)
        L, tau = L.clone(), tau.clone()
        Ln, taun = (None, None) if Ln is None else (Ln.clone(), taun.clone())
        did_split = torch.zeros(len(src), dtype=torch.bool, device=self.dev)
        rows = ((cell >= 0) & (cell < self.n)).all(1).nonzero()[:, 0]
        n, u, rend, cell = n[rows], u[rows], rend[rows], cell[rows]
        step = torch.sign(n)
        face = cell + (n > 0)
        tc = torch.full((len(rows),), r0, dtype=torch.float64, device=self.dev)
        alive = torch.ones(len(rows), dtype=torch.bool, device=self.dev)
        k = 0
        while len(rows):
            t = torch.where(n != 0, (face - u) / torch.where(n != 0, n, torch.ones_like(n)), math.inf)
            tm = t.amin(1)
            ended = rend <= tm
            ds = torch.where(alive, torch.where(ended, rend, tm) - tc, 0.0).clamp(min=0.0)
            seg = ds > 0
            c = torch.where(seg, (cell.long() * self.stride).sum(1), 0)
            x = self.chi[c] * ds
            phi = _phi(x)
            Lr = L[rows]
            xn = Lnr = None
            if Ln is not None:
                xn, Lnr = self.chin[c] * ds, Ln[rows]
            segment(rows, c, n, ds, x, Lr, phi, xn, Lnr)
            L[rows] = Lr * torch.exp(-x)
            tau[rows] = tau[rows] + x
            depth = tau
            if Ln is not None:
                Ln[rows] = Lnr * torch.exp(-xn)
                taun[rows] = taun[rows] + xn
                depth = taun
            drop = seg & (depth[rows] > case["tau_max"])
            did_split[rows] |= alive & ended & ~drop & (rend < cut) & (self.lmax[src[rows]] > l)
            cross = (t - tm[:, None] <= 1e-12 * tm[:, None])
            cell = torch.where(cross, cell + step, cell)
            face = torch.where(cross, face + step, face)
            tc = tm
            alive = alive & ~ended & ~drop & ((cell >= 0) & (cell < self.n)).all(1)
            k += 1
            if k % 8 == 0 or len(rows) < 4096:
                keep = alive.nonzero()[:, 0]
                rows, n, u, rend, cell = rows[keep], n[keep], u[keep], rend[keep], cell[keep]
                step, face, tc, alive = step[keep], face[keep], tc[keep], alive[keep]
        return L, tau, Ln, taun, did_split

    def chunks(self, count, size=1 << 21):
        return [slice(a, min(a + size, count)) for a in range(0, count, size)]

    def forward(self, loss=None):
        """All levels. With ``loss`` (per-segment loss, see ``backward``) the fronts and the
        rays' own losses are kept."""
        case = self.case
        npix = 12 * 4 ** case["level0"]
        src = torch.arange(len(self.L), device=self.dev).repeat_interleave(npix)
        pix = torch.arange(npix, device=self.dev).repeat(len(self.L))
        L, tau = self.L[src] / npix, torch.zeros(len(src), dtype=torch.float64, device=self.dev)
        Ln, taun = (None, None) if self.Ln is None else (self.Ln[src] / npix, tau.clone())
        l, fronts = case["level0"], []
        parent = None

        def pick(t, i):
            return None if t is None else t[i]

        while len(src):
            own = torch.zeros(len(src), dtype=torch.float64, device=self.dev)
            parts = []
            for sl in self.chunks(len(src)):
                def segment(rows, c, n, ds, x, Lr, phi, xn, Lnr):
                    self.G.index_add_(0, c, Lr * ds * phi)
                    dL = Lr * x * phi
                    if loss is not None:
                        own[sl][rows] += loss(c, n, Lr * ds * phi, dL)
                    if xn is not None:
                        dL = dL + Lnr * xn * _phi(xn)
                    if self.F is not None:
                        for a in range(3):
                            self.F[a].index_add_(0, c, dL * n[:, a])
                e = self.walk(l, src[sl], pix[sl], L[sl], tau[sl], pick(Ln, sl), pick(taun, sl), segment)
                i = e[4].nonzero()[:, 0]
                parts.append((i + sl.start, *(pick(t, i) for t in e[:4])))
            if loss is not None:
                fronts.append((l, src, pix, L, tau, own, parent))
            i, eL, etau = (torch.cat([p[k] for p in parts]).repeat_interleave(4) for k in range(3))
            if Ln is not None:
                Ln, taun = (torch.cat([p[k] for p in parts]).repeat_interleave(4) for k in (3, 4))
                Ln = 0.25 * Ln
            four = torch.arange(len(i), device=self.dev) % 4
            src, pix, L, tau, parent = src[i], 4 * pix[i] + four, 0.25 * eL, etau, i
            l += 1
        return fronts

    def outputs(self):
        case, sh = self.case, (int(self.n[2]), int(self.n[1]), int(self.n[0]))
        o = {"gamma": (case["sigma_H"] * self.dx / self.dV * self.G).reshape(sh)}
        if case["force"]:
            o["force"] = (self.F / self.dV).reshape((3,) + sh)
        if case["energy"]:
            o["energy"] = (self.dx / self.dV * self.G).reshape(sh)
        return o

    def backward(self, w, v):
        """Gradients of sum w gamma + sum v . force."""
        gs = self.case["sigma_H"] * self.dx / self.dV
        w = w.double().reshape(-1) * gs
        v = None if v is None else v.double().reshape(3, -1) / self.dV

        def q(c, n):
            return (v[:, c] * n.T).sum(0)

        fronts = self.forward(lambda c, n, G, dL: w[c] * G + (0.0 if v is None else q(c, n) * dL))
        total = [f[5] for f in fronts]
        for k in range(len(fronts) - 1, 0, -1):
            total[k - 1] = total[k - 1].index_add(0, fronts[k][6], total[k])
        grad = torch.zeros_like(self.chi)
        for (l, src, pix, L, tau, _, _), tot in zip(fronts, total):
            for sl in self.chunks(len(src)):
                rem = tot[sl].clone()

                def segment(rows, c, n, ds, x, Lr, phi, xn, Lnr):
                    own = w[c] * Lr * ds * phi
                    d = w[c] * Lr * ds * _dphi(x, phi)
                    if v is not None:
                        own = own + q(c, n) * Lr * x * phi
                        d = d + q(c, n) * Lr * torch.exp(-x)
                    rem[rows] -= own
                    grad.index_add_(0, c, self.chiH[c] * ds * (d - rem[rows]))
                self.walk(l, src[sl], pix[sl], L[sl], tau[sl], None, None, segment)
        dL = torch.zeros_like(self.L).index_add(0, fronts[0][1], total[0]) / self.L
        sh = (int(self.n[2]), int(self.n[1]), int(self.n[0]))
        return grad.reshape(sh), dL


def _xn_exact(gamma, nH, x0, alpha, dt, method):
    g, n, x0 = gamma.double(), nH.double(), x0.double()
    if method == "b":
        a = alpha * n * (1.0 - x0)
        rate = g + a
        xeq = a / torch.where(rate > 0, rate, torch.ones_like(rate))
        x = torch.where(rate > 0, xeq + (x0 - xeq) * torch.exp(-dt * rate), x0)
    else:
        a = alpha * n
        qd = (1.0 - x0) * a * dt
        xeq = 2.0 * a / (g + 2.0 * a + torch.sqrt(g * g + 4.0 * a * g))
        K = torch.exp(-(1.0 / xeq - xeq) * dt * a)
        lit = xeq + (1.0 / xeq - xeq) * (x0 - xeq) * K / ((1.0 / xeq - x0) + (x0 - xeq) * K)
        x = torch.where(g > 0, lit, (x0 + qd) / (1.0 + qd))
    x = x.clamp(0.0, 1.0)
    return {"xn": x, "nH0": x * n}


def exact(case, seed):
    family = case["family"]
    d = _inputs(case, seed)
    if family == "xn":
        return _xn_exact(d["gamma"], d["nH"], d["xn"], d["alpha"], d["dt"], case["method"])
    # a walk in torch costs a few ns per crossing and pass
    if _crossings(case) * (3 if family in ("backward", "autograd") else 1) > 2.5e9:
        return None
    if family == "autograd":
        d["nH0"] = torch.exp(torch.log(d["nH0"]).double())
    t = _Trace64(case, d)
    if family in ("backward", "autograd"):
        grad, dL = t.backward(d["w"], d["v"])
        if family == "backward":
            return {"grad": grad, "dL": dL}
        return {"gamma": t.outputs()["gamma"], "grad": grad, "dL": dL.cpu()}
    t.forward()
    o = t.outputs()
    if family == "trace":
        return o
    gamma, x, nH = o["gamma"], d["nH0"], torch.ones_like(d["nH0"])
    rate = (x.double() * nH.double() * gamma - (nH.double() * (1.0 - x.double())) ** 2).abs()
    dt = 0.1 * torch.where(rate > 0, nH.double() / rate, math.inf).min()
    return {"gamma": gamma, "dt": dt.reshape(1), **_xn_exact(gamma, nH, x, 1.0, dt, "b")}
