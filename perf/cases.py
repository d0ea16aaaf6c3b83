"""Performance cases of the CSEM engine: the runs that modelling, gradient and inversion programs make through
`Engine` and `forward_data`, from the smallest test box to the 256x256x128 towline.

A case is one call (one modelling run, one adjoint run, one gradient, one basis estimate) or, for "autograd", the
forward and backward of one misfit.  Runs are shortened to `nt` steps (the full count of a production run, 35 decay
times, is 6 000 to 20 000): every step costs the same, so the time of a pass scales with nt.

`exact` restates the method in 64 bits with plain torch and numpy (leap-frog Yee or four-point differences, unsplit
CPML, damped transform, basis, gradients); it uses none of the package's code.
"""
import math

import numpy as np
import torch

from paper_2211_16665_gb300.autograd import forward_data
from paper_2211_16665_gb300.engine import Engine
from paper_2211_16665_gb300.workloads import Points

MU0 = 4e-7 * math.pi
F0 = 1.0                  # reference frequency of the correspondence [Hz]
WATER, SEDIMENT = 0.3, 1.0

BASE = {"kind": "data", "cx": 24, "cy": 24, "cz": 24, "st_xy": 0, "st_z": 0, "npml": 10, "h": 50.0, "ratio": 1.05,
        "rho_max": 100.0, "nf": 4, "fmin": 0.25, "fmax": 1.0, "log_f": False, "n_src": 1, "n_rec": 21, "nt": 512,
        "precision": 32, "kahan": 1, "order": 2, "vti": False, "early": 0.0, "budget": 0}

RESERVOIR = {"cx": 80, "cy": 80, "cz": 62, "st_xy": 14, "st_z": 7, "n_rec": 41}           # 128 x 128 x 96
TOWLINE = {"cx": 196, "cy": 196, "cz": 94, "st_xy": 20, "st_z": 7, "n_rec": 64, "n_src": 2}   # 256 x 256 x 128


def listed():
    return [dict(BASE, name=name, **more) for name, more in (
        # the smallest data run: a 40^3 box of the tests, as a line search or a unit test calls it; launches count
        ("box_data", dict(kind="data", cx=24, cy=24, cz=24, npml=8, h=100.0, ratio=1.0, rho_max=20.0, nf=2,
                          fmax=0.75, n_rec=6, nt=600)),
        # one misfit and its gradient on a box of odd sizes (53 x 47 x 43), two sources: a small inversion's iteration
        ("ragged_autograd", dict(kind="autograd", cx=33, cy=27, cz=23, st_xy=2, st_z=2, npml=8, h=100.0,
                                 rho_max=20.0, nf=3, n_src=2, n_rec=7, nt=1000)),
        # the FP64 reference configuration: uniform 68^3, forward with volumes, all of its 1500 steps
        ("uniform_fp64", dict(kind="forward", cx=48, cy=48, cz=48, h=100.0, ratio=1.0, rho_max=2.0, nf=2, fmax=0.75,
                              n_rec=21, nt=1500, precision=64, kahan=0)),
        # forward run of a gradient on the thin-reservoir grid, compensated transform
        ("reservoir_forward", dict(kind="forward", nt=1024, **RESERVOIR)),
        # data modelling with the early end, as the line searches of the inversion call it (full step count)
        ("reservoir_early_data", dict(kind="data", early=1e-6, nt=12328, **RESERVOIR)),
        # fourth-order differences, data run
        ("reservoir_order4", dict(kind="data", order=4, nt=512, **RESERVOIR)),
        # gradient by the time-domain adjoint with checkpoints, VTI medium
        ("vti_time_domain", dict(kind="td", cx=48, cy=44, cz=40, st_xy=4, st_z=2, npml=8, vti=True, n_rec=15, nt=1024,
                                 budget=2 << 30)),
        # four sources per launch on the 116^3 crop of the heterogeneous model, plain FP32 transform, three frequencies
        ("crop_batch", dict(kind="forward", cx=76, cy=76, cz=84, st_xy=10, st_z=6, nf=3, n_src=4, n_rec=64, kahan=0,
                            nt=512)),
        # the towline's two runs of a gradient, two sources per launch: the production size
        ("towline_forward", dict(kind="forward", nt=256, **TOWLINE)),
        ("towline_adjoint", dict(kind="adjoint", nt=256, **TOWLINE)),
        # the cell gradient from two runs' volumes at that size
        ("towline_gradient", dict(kind="gradient", nt=256, **TOWLINE)),
        # the adjoint-source basis of eight frequencies over a full run (0.1 to 1.5 Hz, 19 492 steps)
        ("basis_eight", dict(kind="basis", npml=8, nf=8, fmin=0.1, fmax=1.5, log_f=True, nt=19492)),
    )]


def draw(rng):
    kind = rng.choice(["data", "forward", "forward", "adjoint", "autograd", "td", "gradient", "basis"])
    c = dict(BASE, kind=kind)
    c["nf"] = rng.randint(1, 8) if kind in ("forward", "basis") else rng.randint(1, 5)
    c["fmin"], c["fmax"] = round(rng.uniform(0.1, 0.25), 3), round(rng.uniform(0.75, 1.5), 3)
    c["log_f"] = rng.random() < 0.5
    c["npml"] = rng.choice([6, 8, 10])
    if kind == "basis":
        c["nt"] = int(round(math.exp(rng.uniform(math.log(600), math.log(19492)))))
        return c
    c["precision"] = 64 if kind != "td" and rng.random() < 0.15 else 32
    c["kahan"] = int(c["precision"] == 32 and rng.random() < 0.7)
    c["order"] = 4 if kind in ("data", "forward", "adjoint") and rng.random() < 0.2 else 2
    c["vti"] = rng.random() < 0.2
    c["early"] = 1e-6 if kind == "data" and c["order"] == 2 and rng.random() < 0.3 else 0.0
    c["n_src"] = rng.choice([1, 1, 2, 3, 4])
    c["n_rec"] = rng.randint(4, 64)
    c["st_xy"], c["st_z"] = rng.randint(0, 14), rng.randint(0, 7)
    c["rho_max"] = rng.choice([20.0, 100.0])
    # core sizes: the geometric mean over its whole range, the axes within a factor of about two
    slow = c["precision"] == 64 or kind == "td" or c["early"] > 0
    side = math.exp(rng.uniform(math.log(14), math.log(50 if slow else 130)))
    for axis in ("cx", "cy", "cz"):
        c[axis] = max(12, int(round(side * rng.uniform(0.7, 1.35))))
    if rng.random() < 0.5:       # half of the grids have even sizes along x, as configurations have; the rest any
        c["cx"] += c["cx"] % 2
    cells = float(np.prod(shape(c)))
    c["n_src"] = max(1, min(c["n_src"], int(1.7e7 / cells)))
    if kind == "td":
        c["n_src"] = min(c["n_src"], 2)
        c["nt"] = int(min(rng.randint(200, 1000), 1.2e9 / (cells * c["n_src"])))
        c["budget"] = 4 << 30
    else:
        share = {"autograd": 0.4}.get(kind, 0.9) * (0.1 if c["precision"] == 64 else 0.5 if c["order"] == 4 else 1.0)
        most = share * 4.3e9 / (cells * c["n_src"])
        c["nt"] = int(max(64, min(math.exp(rng.uniform(math.log(256), math.log(2000))), most)))
        if c["early"]:
            c["nt"] = 4000
    return c


# -- inputs ----------------------------------------------------------------------------------------------------------

def axis_nodes(n_core, n_st, npml, h, ratio, start):
    """Node coordinates: n_core cells of width h from `start`, n_st cells growing by `ratio` and npml of the last width on each side."""
    grow = [h * ratio ** (m + 1) for m in range(n_st)]
    grow += [grow[-1] if grow else h] * npml
    widths = grow[::-1] + [h] * n_core + grow
    return start - sum(grow) + np.concatenate([[0.0], np.cumsum(widths)])


def grid(c):
    xn = axis_nodes(c["cx"], c["st_xy"], c["npml"], c["h"], c["ratio"], -0.5 * c["h"] * c["cx"])
    yn = axis_nodes(c["cy"], c["st_xy"], c["npml"], c["h"], c["ratio"], -0.5 * c["h"] * c["cy"])
    zn = axis_nodes(c["cz"], c["st_z"], c["npml"], c["h"], c["ratio"], 0.0)
    return xn, yn, zn


def shape(c):
    pad = 2 * c["npml"]
    return c["cz"] + 2 * c["st_z"] + pad, c["cy"] + 2 * c["st_xy"] + pad, c["cx"] + 2 * c["st_xy"] + pad


def freqs_of(c, seed):
    """The survey's frequencies [Hz]; another seed is another survey."""
    scale = 1.0 + 1e-3 * (seed % 29)
    if c["nf"] == 1:
        return np.array([scale * c["fmax"]])
    f = np.geomspace(c["fmin"], c["fmax"], c["nf"]) if c["log_f"] else np.linspace(c["fmin"], c["fmax"], c["nf"])
    return scale * f


def real_of(c):
    return torch.float32 if c["precision"] == 32 else torch.float64


def generator(seed, device, salt):
    return torch.Generator(device=device).manual_seed(1_000_003 * salt + seed)


def model(c, seed, device):
    """Water over sediment with cell-to-cell scatter, and a resistive slab below the seabed; (rho_h, rho_v) for VTI."""
    xn, yn, zn = grid(c)
    mid = [torch.as_tensor(0.5 * (a[1:] + a[:-1]), device=device) for a in (zn, yn, xn)]
    z, y, x = torch.meshgrid(*mid, indexing="ij")
    g = generator(seed, device, 1)
    seabed = c["h"] * (c["cz"] // 3)
    scatter = torch.exp(0.2 * torch.randn(z.shape, generator=g, device=device, dtype=torch.float64))
    rho = torch.where(z < seabed, torch.full_like(z, WATER), SEDIMENT * scatter)
    slab = (x.abs() < 0.3 * c["h"] * c["cx"]) & (y.abs() < 0.3 * c["h"] * c["cy"]) & \
        (z >= seabed + 4 * c["h"]) & (z < seabed + 6 * c["h"])
    rho = torch.where(slab, torch.full_like(z, 0.9 * c["rho_max"]), rho).clamp(max=c["rho_max"])
    if c["vti"]:
        rho = torch.stack([rho, torch.where(z < seabed, rho, 2.0 * rho).clamp(max=c["rho_max"])])
    return rho.to(real_of(c)).contiguous()


def points(c, seed):
    """x-dipoles half a cell above the seabed, and receivers on it, at positions drawn from the seed: (sources, receivers) as (xyz, component)."""
    r = np.random.default_rng(seed)
    seabed, h = c["h"] * (c["cz"] // 3), c["h"]
    half = 0.5 * h * c["cx"] - 2 * h
    xs = np.linspace(-0.5, 0.5, c["n_src"] + 2)[1:-1] * 2 * half * 0.6
    src = [(x + r.uniform(-h, h), r.uniform(-h, h), seabed - 0.5 * h) for x in xs]
    side = int(math.ceil(math.sqrt(c["n_rec"])))
    hy = 0.5 * h * c["cy"] - 2 * h
    at = [(x, y) for y in np.linspace(-hy, hy, side) for x in np.linspace(-half, half, side)][:c["n_rec"]]
    rec = [(x + r.uniform(-0.4, 0.4) * h, y + r.uniform(-0.4, 0.4) * h, seabed) for x, y in at]
    return (np.array(src), np.zeros(len(src), np.int32)), (np.array(rec), r.integers(0, 2, len(rec)).astype(np.int32))


def observed(c, src, rec, seed):
    """Data of the size that a survey sees: the dipole field of a whole space of 1 ohm-m, with 5 % scatter."""
    r = np.random.default_rng(seed + 7)
    d = rec[0][None, :, :] - src[0][:, None, :]
    rr = np.sqrt((d ** 2).sum(-1)) + c["h"]
    k = np.sqrt(1j * 2 * np.pi * freqs_of(c, seed) * MU0 / SEDIMENT)
    kr = rr[..., None] * k
    along = (d[..., 0] * np.take_along_axis(d, rec[1][None, :, None].astype(int), -1)[..., 0] / rr ** 2)[..., None]
    same = (rec[1] == 0)[None, :, None]
    e = SEDIMENT / (4 * np.pi * rr[..., None] ** 3) * np.exp(1j * kr) * ((3 - 3j * kr - kr ** 2) * along +
                                                                  same * (kr ** 2 + 1j * kr - 1))
    return e * (1 + 0.05 * (r.standard_normal(e.shape) + 1j * r.standard_normal(e.shape)))


def volume(c, seed, salt, n_src, vol_shape, dtype, device):
    """A transform volume as a run leaves it: smooth decay away from the middle, zero on the outer faces and off the lattice."""
    nz, ny, nx = shape(c)
    g = generator(seed, device, salt)
    v = torch.randn(vol_shape, generator=g, device=device, dtype=dtype)
    for a, n in ((3, nz), (4, ny), (5, nx)):
        t = torch.linspace(-1, 1, n + 1, device=device)
        w = torch.zeros(vol_shape[a], device=device)
        w[:n + 1] = 1e-6 * torch.exp(-4 * t.abs())
        v *= w.view([-1 if b == a else 1 for b in range(6)]).to(real_of(c))
    for comp, a in ((0, 3), (0, 4), (1, 3), (1, 5), (2, 4), (2, 5)):     # tangential components are zero on the outer faces
        n = {3: nz, 4: ny, 5: nx}[a]
        v[:, comp].select(a - 1, 0).zero_()
        v[:, comp].select(a - 1, n).zero_()
    for comp, a in ((0, 5), (1, 4), (2, 3)):                             # half nodes: one entry fewer along the component's axis
        v[:, comp].select(a - 1, {3: nz, 4: ny, 5: nx}[a]).zero_()
    return v


def make_points(p):
    return Points.make(p[0], p[1])


def prepare(case, seed):
    c = dict(BASE, **case)
    dev = torch.device("cuda")
    xn, yn, zn = grid(c)
    steps = c["kind"] not in ("gradient", "basis")         # these two run no time step, so there is no launch to tune
    eng = Engine(xn, yn, zn, c["npml"], freqs_of(c, seed), f0=F0, rho_max=c["rho_max"], precision=c["precision"],
                 kahan=c["kahan"], max_src=c["n_src"], max_rec=c["n_rec"], nt=c["nt"], autotune=steps, vti=c["vti"],
                 order=c["order"], ring_slots=0 if steps else 17)
    s = {"case": c, "eng": eng}
    if c["kind"] == "basis":
        return s
    s["rho"] = model(c, seed, dev)
    src, rec = points(c, seed)
    s["src"], s["rec"] = make_points(src), make_points(rec)
    if c["early"]:
        eng.set_early_stop(c["early"])
    if c["kind"] in ("adjoint", "td", "autograd"):
        s["obs"] = torch.as_tensor(observed(c, src, rec, seed), device=dev)
    if c["kind"] in ("adjoint", "autograd"):
        s["basis"], _, _ = eng.estimate_adjoint_basis(fit_target=1e-3)
    if c["kind"] == "autograd":
        s["ln_rho"] = torch.log(s["rho"].to(torch.float64))
    if c["kind"] == "gradient":
        vs = eng.volume_shape(c["n_src"])
        s["E"] = volume(c, seed, 2, c["n_src"], vs, eng.cplx, dev)
        s["V"] = volume(c, seed, 3, c["n_src"], vs, eng.cplx, dev)
    return s


def run(s):
    """One call.  The spectra of an FP32 engine are kept in complex64, as a program keeps them beside its FP32 volumes
    and gradients: the field they are sums of is stepped in FP32."""
    c, eng = s["case"], s["eng"]
    kind = c["kind"]
    if kind == "data":
        return {"data": eng.fwd_model(s["rho"], s["src"], s["rec"]).to(eng.cplx)}
    if kind == "forward":
        d, vol = eng.fwd_model(s["rho"], s["src"], s["rec"], keep_volume=True)
        return {"data": d.to(eng.cplx), "volume": vol}
    if kind == "adjoint":
        return {"volume": eng.adjoint_model(s["rho"], s["rec"], s["obs"], s["basis"])}
    if kind == "gradient":
        return {"gradient": eng.gradient(s["rho"], s["E"], s["V"])}
    if kind == "td":
        return {"gradient": eng.gradient_td(s["rho"], s["src"], s["rec"], s["obs"], budget_bytes=c["budget"])}
    if kind == "basis":
        return {"basis": eng.estimate_adjoint_basis(fit_target=1e-3)[0]}
    ln_rho = s["ln_rho"].detach().requires_grad_(True)
    d = forward_data(ln_rho, eng, s["src"], s["rec"], s["basis"])
    res = s["obs"] - d
    (0.5 * torch.sum(res.real ** 2 + res.imag ** 2)).backward()
    return {"data": d.detach().to(eng.cplx), "gradient": ln_rho.grad.to(real_of(c))}


def work(case):
    """Each step reads and writes the six field components of every cell once; model, volumes and gradient move once."""
    c = dict(BASE, **case)
    nz, ny, nx = shape(c)
    cells, r, S, nf, nt = nx * ny * nz, c["precision"] // 8, c["n_src"], c["nf"], c["nt"]
    models = cells * r * (2 if c["vti"] else 1)
    vol = S * 3 * nf * cells * 2 * r
    step_b, step_f = 12 * r * cells * S, (36 if c["order"] == 2 else 84) * cells * S
    dft_f = S * 3 * nf * cells * 4
    kind = c["kind"]
    if kind == "basis":
        return {"bytes": 16 * nf * nt, "flops": 2 * nf * (2 * nf + 1) * nt * 8 * nf}
    if kind == "gradient":
        return {"bytes": 2 * vol + 2 * models, "flops": 4 * S * 3 * nf * cells}
    if kind == "data":
        n = nt // 2 if c["early"] else nt
        return {"bytes": models + n * step_b, "flops": n * step_f}
    if kind in ("forward", "adjoint"):
        return {"bytes": models + vol + nt * step_b, "flops": nt * (step_f + dft_f)}
    if kind == "td":
        return {"bytes": 2 * models + 2 * nt * step_b, "flops": nt * (2 * step_f + 9 * cells * S)}
    return {"bytes": 2 * models + 2 * nt * step_b, "flops": 2 * nt * (step_f + dft_f)}


# -- the same in 64 bits ---------------------------------------------------------------------------------------------

class Exact:
    """The discretisation in FP64: fields are [source, nz+1, ny+1, nx+1] on the node lattice, Ex at (i+1/2, j, k) and so on."""

    def __init__(self, c, seed, rho, device):
        self.c, self.dev = c, device
        self.nodes = grid(c)                                             # x, y, z
        self.n = [a.size - 1 for a in self.nodes]
        self.freqs = freqs_of(c, seed)
        self.w0 = 2 * np.pi * F0
        self.a = np.sqrt(2 * np.pi * self.freqs * self.w0)
        self.k = np.sqrt(-1j * 2 * np.pi * self.freqs / (2 * self.w0))
        v = math.sqrt(2 * self.w0 * c["rho_max"] / MU0)
        self.h = [np.diff(a) for a in self.nodes]
        self.ht = [np.concatenate([[0.5 * h[0]], 0.5 * (h[:-1] + h[1:]), [0.5 * h[-1]]]) for h in self.h]
        self.wh, self.wn = zip(*(self._weights(a) for a in range(3)))
        if c["order"] == 4:
            s2 = 0.0
            for a in range(3):
                rh, rn = np.abs(self.wh[a]).sum(1), np.abs(self.wn[a]).sum(1)
                s2 += np.maximum(rh, np.maximum(rn[:-1], rn[1:])).max() ** 2
            self.dt = 0.99 * 2 / (v * math.sqrt(s2))
        else:
            self.dt = 0.99 / (v * math.sqrt(sum((1 / h ** 2).max() for h in self.h)))
        self.tabs = []
        for a in range(3):
            half = 0.5 * (self.nodes[a][1:] + self.nodes[a][:-1])
            self.tabs.append({"h": (self.wh[a], *self._cpml(a, half, v)), "n": (self.wn[a], *self._cpml(a, self.nodes[a], v))})
        self.rho = rho.to(torch.float64)
        self.cE = 2 * self.w0 * self.dt * self._edge_average()

    def _weights(self, a):
        x, h, ht, n = self.nodes[a], self.h[a], self.ht[a], self.n[a]
        wh, wn = np.zeros((n, 4)), np.zeros((n + 1, 4))
        wh[:, 1], wh[:, 2] = -1 / h, 1 / h
        wn[1:-1, 1], wn[1:-1, 2] = -1 / ht[1:-1], 1 / ht[1:-1]
        if self.c["order"] == 4:
            def fit(at, xs):
                d = xs - at
                scale = np.abs(d).max()
                return np.linalg.solve(np.vander(d / scale, 4, increasing=True).T, [0.0, 1.0, 0.0, 0.0]) / scale
            xh = 0.5 * (x[1:] + x[:-1])
            for p in range(1, n - 1):
                wh[p] = fit(xh[p], x[p - 1:p + 3])
            for q in range(2, n - 1):
                wn[q] = fit(x[q], xh[q - 2:q + 2])
        return wh, wn

    def _cpml(self, a, p, v):
        x, npml, n = self.nodes[a], self.c["npml"], self.n[a]
        b, c = np.zeros_like(p), np.zeros_like(p)
        for edge, out, L in ((x[npml], -1, x[npml] - x[0]), (x[n - npml], 1, x[n] - x[n - npml])):
            xi = out * (p - edge)
            m = xi > 0
            d = -3 * v * math.log(1e-6) / (2 * L) * (xi[m] / L) ** 2
            al = math.pi * F0 * (1 - xi[m] / L)
            b[m] = np.exp(-(d + al) * self.dt)
            c[m] = d * (b[m] - 1) / (d + al)
        return b, c

    def _vol(self):
        h = [torch.as_tensor(a, device=self.dev) for a in self.h]
        return h[2][:, None, None] * h[1][None, :, None] * h[0][None, None, :]

    @staticmethod
    def _edge_sum(A, comp):
        P = torch.nn.functional.pad(A, (1, 1, 1, 1, 1, 1))
        ax = {0: (0, 1), 1: (0, 2), 2: (1, 2)}[comp]                    # array axes that are averaged over
        for a in ax:
            n = P.shape[a]
            P = P.narrow(a, 0, n - 1) + P.narrow(a, 1, n - 1)
        own = 2 - comp
        n = P.shape[own]                                                # cells 0 .. n-1 of the component's own axis, and one zero
        return P.narrow(own, 1, n - 1)

    def _edge_average(self):
        V = self._vol()
        out = []
        for comp in range(3):
            r = self.rho if self.rho.dim() == 3 else self.rho[1 if comp == 2 else 0]
            num, den = self._edge_sum(V / r, comp), self._edge_sum(V, comp)
            out.append(torch.where(num > 0, den / num.clamp(min=1e-300), torch.zeros_like(num)))
        E = torch.stack(out)
        for comp, a in ((0, 1), (0, 2), (1, 1), (1, 3), (2, 2), (2, 3)):     # no update on the outer faces
            E[comp].select(a - 1, 0).zero_()
            E[comp].select(a - 1, E.shape[a] - 1).zero_()
        return E

    def taps(self, pts, inject):
        """(point, component, flat lattice index, weight) of trilinear interpolation, or of its transpose over the dual volume."""
        out = []
        N = [n + 1 for n in self.n]
        for q, (xyz, comp) in enumerate(zip(*pts)):
            ax = []
            for a in range(3):
                g = 0.5 * (self.nodes[a][1:] + self.nodes[a][:-1]) if a == comp else self.nodes[a]
                m = int(np.clip(np.searchsorted(g, xyz[a], side="right") - 1, 0, g.size - 2))
                t = (xyz[a] - g[m]) / (g[m + 1] - g[m])
                ax.append(((m, 1 - t), (m + 1, t)))
            for i, wi in ax[0]:
                for j, wj in ax[1]:
                    for k, wk in ax[2]:
                        w = wi * wj * wk
                        if inject:
                            w /= np.prod([(self.h if a == comp else self.ht)[a][p] for a, p in enumerate((i, j, k))])
                        out.append((q, int(comp), (k * N[1] + j) * N[0] + i, w))
        q, comp, idx, w = zip(*out)
        t = lambda v, d: torch.as_tensor(np.array(v), dtype=d, device=self.dev)  # noqa: E731
        return t(q, torch.int64), t(comp, torch.int64), t(idx, torch.int64), t(w, torch.float64)

    def _derivative(self, f, a, at):
        """d f / d(axis a) at the half nodes ("h": from nodes) or at the nodes ("n": from half nodes, zero on the outer ones)."""
        dim = 3 - a
        n = self.n[a]
        w = self.dw[a][at]
        if self.c["order"] == 2:
            d = f.narrow(dim, 1, n) - f.narrow(dim, 0, n) if at == "h" else f.narrow(dim, 1, n - 1) - f.narrow(dim, 0, n - 1)
            return d.mul_(w[2] if at == "h" else w[2].narrow(dim, 1, n - 1))
        m = n if at == "h" else n - 1
        first = -1                          # f index of tap 0 at output 0 ("h": node -1 at half node 0; "n": half node -1 at node 1)
        length = n + 1 if at == "h" else n
        d = None
        for t in range(4):
            lo, hi = first + t, first + t + m
            wt = w[t] if at == "h" else w[t].narrow(dim, 1, m)
            c0, c1 = max(0, -lo), max(0, hi - length)
            if d is None:
                d = torch.zeros([m if x == dim else s for x, s in enumerate(f.shape)], dtype=f.dtype, device=f.device)
            k = m - c0 - c1
            d.narrow(dim, c0, k).addcmul_(f.narrow(dim, lo + c0, k), wt.narrow(dim, c0, k))
        return d

    def start(self, S):
        nz, ny, nx = self.n[2], self.n[1], self.n[0]
        self.dw, self.ba = [], []
        for a in range(3):
            v = [1, 1, 1, 1]
            v[3 - a] = -1
            col = lambda x: torch.as_tensor(np.ascontiguousarray(x), device=self.dev).view(v)  # noqa: E731
            self.dw.append({at: [col(self.tabs[a][at][0][:, t]) for t in range(4)] for at in "hn"})
            self.ba.append({at: (col(self.tabs[a][at][1]), col(self.tabs[a][at][2])) for at in "hn"})
        z = lambda: torch.zeros((S, nz + 1, ny + 1, nx + 1), dtype=torch.float64, device=self.dev)  # noqa: E731
        return {"E": torch.stack([z(), z(), z()]), "H": [z(), z(), z()], "psi": {}}

    def _stretched(self, st, key, f, a, at):
        d = self._derivative(f, a, at)
        dim, n, p = 3 - a, d.shape[3 - a], self.c["npml"]
        b, c = self.ba[a][at]
        if at == "n":
            b, c = b.narrow(dim, 1, n), c.narrow(dim, 1, n)
        for side, lo in ((0, 0), (1, n - p)):                            # the recursion acts in the outer npml cells only
            if p == 0:
                break
            ds = d.narrow(dim, lo, p)
            q = st["psi"].get((key, side))
            if q is None:
                q = st["psi"][(key, side)] = torch.zeros_like(ds)
            q.mul_(b.narrow(dim, lo, p)).addcmul_(ds, c.narrow(dim, lo, p))
            ds.add_(q)
        return d

    def step(self, st):
        """E^n, H^{n-1/2} -> H^{n+1/2}, E^{n+1} (without the source)."""
        nx, ny, nz = self.n
        ex, ey, ez = st["E"]
        hx, hy, hz = st["H"]
        cH = self.dt / MU0
        Z, Y, X = slice(0, nz), slice(0, ny), slice(0, nx)
        D = lambda key, f, a, at: self._stretched(st, key, f, a, at)  # noqa: E731
        hx[:, Z, Y, :] -= cH * (D("hx1", ez[:, Z], 1, "h") - D("hx2", ey[:, :, Y], 2, "h"))
        hy[:, Z, :, X] -= cH * (D("hy1", ex[..., X], 2, "h") - D("hy2", ez[:, Z], 0, "h"))
        hz[:, :, Y, X] -= cH * (D("hz1", ey[:, :, Y], 0, "h") - D("hz2", ex[..., X], 1, "h"))
        iz, iy, ix = slice(1, nz), slice(1, ny), slice(1, nx)
        c = self.cE
        ex[:, iz, iy, X] += c[0][iz, iy, X] * (D("ex1", hz[:, iz, :, X][:, :, Y], 1, "n") - D("ex2", hy[:, Z, iy, X], 2, "n"))
        ey[:, iz, Y, ix] += c[1][iz, Y, ix] * (D("ey1", hx[:, Z, Y, ix], 2, "n") - D("ey2", hz[:, iz, Y, X], 0, "n"))
        ez[:, Z, iy, ix] += c[2][Z, iy, ix] * (D("ez1", hy[:, Z, iy, X], 0, "n") - D("ez2", hx[:, Z, Y, ix], 1, "n"))

    def inject(self, st, taps, amp):
        """amp [source, point]: the moments of J' at this step."""
        q, comp, idx, w = taps
        S = amp.shape[0]
        flat = st["E"].view(3, S, -1)
        add = -self.cE.view(3, -1)[comp, idx] * w * amp[:, q]            # [S, taps]
        for s in range(S):
            flat.index_put_((comp, torch.full_like(comp, s), idx), add[s], accumulate=True)

    def weights(self, nt):
        t = np.arange(nt)[:, None] * self.dt
        return np.exp((-1 + 1j) * self.a * t)                            # [nt, nf]

    def simulate(self, S, nt, moments, inj, rec=None, vol=False, keep=False, early=0.0):
        """moments(n) -> [S, point] or None.  Returns the receiver and volume transforms, and the E of every step (keep)."""
        st = self.start(S)
        w = torch.as_tensor(self.weights(nt), device=self.dev)
        nf = w.shape[1]
        R = None if rec is None else torch.zeros((S, self.c["n_rec"], nf), dtype=torch.complex128, device=self.dev)
        N = st["E"].numel()
        acc = torch.zeros((2 * nf, N), dtype=torch.float64, device=self.dev) if vol else None
        M = 16
        snap = torch.empty((M, N), dtype=torch.float64, device=self.dev) if vol else None
        kept, last, filled, n0 = [], None, 0, 0
        tr = []
        for n in range(nt):
            if vol:
                snap[filled] = st["E"].view(-1)
                filled += 1
                if filled == M or n == nt - 1:
                    ww = torch.cat([w[n0:n + 1].real, w[n0:n + 1].imag], 1)
                    acc.addmm_(ww.t().contiguous(), snap[:filled])
                    filled, n0 = 0, n + 1
            if keep:
                kept.append(st["E"].clone())
            if rec is not None:
                q, comp, idx, tw = rec
                val = st["E"].view(3, S, -1)[comp, :, idx].t() * tw     # [S, taps]
                tr.append(torch.zeros((S, self.c["n_rec"]), dtype=torch.float64, device=self.dev).index_add_(1, q, val))
                if len(tr) == 64 or n == nt - 1:
                    block = torch.stack(tr)
                    R = R + torch.einsum("nsr,nf->srf", block.to(torch.complex128), w[n + 1 - len(tr):n + 1])
                    tr = []
                    if early and (n + 1) % 64 == 0:
                        if last is not None and bool(((R - last).abs() <= early * R.abs()).all()):
                            break
                        last = R
            self.step(st)
            m = moments(n)
            if m is not None:
                self.inject(st, inj, m)
        if keep:
            kept.append(st["E"].clone())
        if vol:
            shp = (nf,) + tuple(st["E"].shape)
            acc = torch.complex(acc[:nf].reshape(shp), acc[nf:].reshape(shp))   # [nf, 3, S, nz+1, ny+1, nx+1]
        return R, acc, kept

    def forward(self, src, rec, nt, **kw):
        S = len(src[0])
        one = torch.eye(S, dtype=torch.float64, device=self.dev) / self.dt
        alpha = self.k * self.dt / np.exp((-1 + 1j) * self.a * 0.5 * self.dt)
        R, V, kept = self.simulate(S, nt, lambda n: one if n == 0 else None, self.taps(src, True), self.taps(rec, False), **kw)
        al = torch.as_tensor(alpha, device=self.dev)
        return R * al, (None if V is None else V * al.view(-1, 1, 1, 1, 1, 1)), kept

    def basis(self, nt, fit_target):
        t = (np.arange(nt) + 0.5) * self.dt
        z = np.exp((-1 + 1j) * self.a[:, None] * t)
        B = np.concatenate([z.real, z.imag])
        U, s, Vt = np.linalg.svd(B, full_matrices=False)
        gamma = 1e-12
        while True:
            g = gamma * s[0] ** 2
            P = (Vt.T * (s / (s ** 2 + g))) @ U.T
            fit = np.abs((U * (s ** 2 / (s ** 2 + g))) @ U.T - np.eye(B.shape[0])).max()
            if fit <= fit_target or gamma <= 1.0001e-16:
                return P
            gamma = max(gamma / 100, 1e-16)

    def adjoint(self, rec, resid, nt):
        """resid [S, R, nf] complex: conj(v) on every edge, from the receivers driven by the basis series of conj(resid)."""
        B = torch.as_tensor(self.basis(nt, 1e-3), device=self.dev)
        cc = torch.as_tensor(self.k, device=self.dev) * resid.conj() / self.dt
        cc = torch.cat([cc.real, cc.imag], 2)
        _, V, _ = self.simulate(resid.shape[0], nt, lambda n: cc @ B[n], self.taps(rec, True), vol=True)
        return V * self.dt

    def to_cells(self, p):
        """p [3, nz+1, ny+1, nx+1] on the edges -> the gradient in ln rho on the cells."""
        nx, ny, nz = self.n
        parts = []
        for comp in range(3):
            q = p[comp]
            for a in {0: (0, 1), 1: (0, 2), 2: (1, 2)}[comp]:
                n = q.shape[a]
                q = q.narrow(a, 0, n - 1) + q.narrow(a, 1, n - 1)
            parts.append(q.narrow(2 - comp, 0, self.n[comp]))
        V = 0.25 * self._vol()
        if self.rho.dim() == 4:
            return torch.stack([-V * (parts[0] + parts[1]) / self.rho[0], -V * parts[2] / self.rho[1]])
        return -V * (parts[0] + parts[1] + parts[2]) / self.rho

    def gradient(self, E, V):
        return self.to_cells(-(E * V).real.sum(dim=(0, 2)))

    def gradient_td(self, src, rec, resid, nt):
        alpha = self.k * self.dt / np.exp((-1 + 1j) * self.a * 0.5 * self.dt)
        _, _, E = self.forward(src, rec, nt, keep=True)
        w = torch.as_tensor(self.weights(nt) * alpha, device=self.dev)
        q = torch.einsum("srf,nf->nsr", resid.conj(), w).real
        st = self.start(resid.shape[0])
        inj = self.taps(rec, True)
        p = torch.zeros_like(st["E"][:, 0])
        for m in range(nt):
            p += (st["E"] * (E[nt - m] - E[nt - 1 - m])).sum(1)
            self.step(st)
            self.inject(st, inj, q[nt - 1 - m])
        return self.to_cells(-p / (2 * self.w0 * self.dt))


def padded(V, pitch, c):
    """[nf, 3, S, z, y, x] -> the engine's [S, 3, nf, z, y, pitch]."""
    V = V.permute(2, 1, 0, 3, 4, 5)
    out = torch.zeros(tuple(V.shape[:5]) + (pitch,), dtype=V.dtype, device=V.device)
    out[..., :V.shape[5]] = V
    return out


def exact(case, seed):
    c = dict(BASE, **case)
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    nz, ny, nx = shape(c)
    pitch = (nx + 8) // 8 * 8
    cells = nx * ny * nz
    kind = c["kind"]
    if kind == "basis":
        return {"basis": torch.as_tensor(Exact(c, seed, torch.ones(shape(c), device=dev), dev).basis(c["nt"], 1e-3))}
    if cells * c["n_src"] * c["nt"] > 2e10:
        return None
    src, rec = points(c, seed)
    rho = model(c, seed, dev)
    x = Exact(c, seed, rho, dev)
    if kind in ("data", "forward"):
        d, V, _ = x.forward(src, rec, c["nt"], vol=kind == "forward", early=c["early"] if kind == "data" else 0.0)
        return {"data": d} if kind == "data" else {"data": d, "volume": padded(V, pitch, c)}
    if kind == "gradient":
        vs = (c["n_src"], 3, c["nf"], nz + 1, ny + 1, pitch)
        dtype = torch.complex64 if c["precision"] == 32 else torch.complex128
        E, V = (volume(c, seed, salt, c["n_src"], vs, dtype, dev)[..., :nx + 1] for salt in (2, 3))
        p = torch.zeros((3, nz + 1, ny + 1, nx + 1), dtype=torch.float64, device=dev)
        for s in range(c["n_src"]):
            for f in range(c["nf"]):
                p -= (E[s, :, f].to(torch.complex128) * V[s, :, f].to(torch.complex128)).real
        return {"gradient": x.to_cells(p)}
    obs = torch.as_tensor(observed(c, src, rec, seed), device=dev)
    if kind == "adjoint":
        return {"volume": padded(x.adjoint(rec, obs, c["nt"]), pitch, c)}
    if kind == "td":
        return {"gradient": x.gradient_td(src, rec, obs, c["nt"])}
    ln_rho = torch.log(rho.to(torch.float64))
    x = Exact(c, seed, torch.exp(ln_rho).to(real_of(c)), dev)
    d, E, _ = x.forward(src, rec, c["nt"], vol=True)
    V = x.adjoint(rec, obs - d, c["nt"])
    return {"data": d, "gradient": x.gradient(E, V)}
