"""Workloads of the collision operator, the transport step and the IMEX steps for timing and comparison.

listed() names the cases, draw() gives more of the same ranges, prepare() makes a program's state before the call,
run() is one call of the public entry points, work() counts what a pass cannot do without, and exact() computes what
run() returns in 64 bits with plain torch and numpy.
"""
import functools
import math

import numpy as np
import torch

from paper_2103_14890_gb300 import binding as bz
from paper_2103_14890_gb300 import workloads

FULL = {"dim": 2, "N": 32, "L": 10.0, "gamma": 1.0, "dirs": 0, "conserve": False}
MESH = {"mesh": "sod", "size": 100, "N": 32, "L": 10.0}


def listed():
    return [
        # a homogeneous relaxation test (BKW, Sec. 4.1: 16^2 velocities, Maxwell molecules) on a few cells: launch latency
        {**FULL, "name": "collide-16-64", "kind": "collide", "N": 16, "L": 8.0, "gamma": 0.0, "precision": "fp32",
         "cells": 64, "input": "bi"},
        # the collision operator over a large mesh, hard spheres, shocks: the framework's headline workload
        {**FULL, "name": "collide-32-65536", "kind": "collide", "precision": "fp32", "cells": 65536,
         "input": "shifted"},
        # reference-accuracy runs of the same operator on noisy data, a batch that is no multiple of any tile
        {**FULL, "name": "collide-32-fp64", "kind": "collide", "precision": "fp64", "cells": 4099, "input": "noisy"},
        # noisy data whose gain and loss cancel: FP32 arrays, double-float mode sum, with the conservation fix
        {**FULL, "name": "collide-32-fp32x2", "kind": "collide", "precision": "fp32x2", "cells": 4096,
         "input": "noisy", "conserve": True},
        # three velocity dimensions, the largest 3-D grid
        {**FULL, "name": "collide-3d-16", "kind": "collide", "dim": 3, "N": 16, "precision": "fp32", "cells": 1000,
         "input": "bi"},
        # the finest 2-D grid (the last row of the spectral convergence table of Sec. 4.1)
        {**FULL, "name": "collide-64", "kind": "collide", "N": 64, "gamma": 0.0, "precision": "fp32", "cells": 500,
         "input": "bi"},
        # independent simulations with their own grids in one call (16^2 to 48^2 and 16^3)
        {"name": "group-mixed", "kind": "group", "precision": "fp32",
         "instances": "2:16:6983 2:24:16515 2:16:3781 2:48:40256 2:24:1949 2:48:13632 2:32:6966 2:48:5748 "
                      "3:16:1000 3:16:1000"},
        # the fast spectral form (Maxwell molecules, eight directions) on one mesh's cells
        {**FULL, "name": "fast-32", "kind": "collide", "gamma": 0.0, "dirs": 8, "precision": "fp32", "cells": 19802,
         "input": "shifted"},
        # distributions that live in page-locked host memory
        {**FULL, "name": "host-32", "kind": "host", "precision": "fp32", "cells": 32768, "input": "shifted"},
        # third-order transport of the explosion problem (Sec. 4.2) on its triangle mesh
        {**MESH, "name": "transport-tri-o3", "kind": "transport", "order": 3, "precision": "fp32"},
        # a full second-order step of the explosion problem: transport, hard-sphere collisions, ARS(2,2,2)
        {**MESH, "name": "step-tri", "kind": "step", "order": 2, "precision": "fp32", "scheme": "ars222",
         "model": "boltzmann", "gamma": 1.0, "dirs": 0, "eps": 5e-3, "conserve": False},
        # a third-order step of the vortex study in the fluid limit on the paper's polygonal meshes, 30^2 velocities
        {"name": "vortex-voronoi-o3", "kind": "step", "mesh": "voronoi", "size": 2603, "N": 30, "L": 10.0, "order": 3,
         "precision": "fp64", "scheme": "bpr343", "model": "bgk", "gamma": 0.0, "dirs": 0, "eps": 1e-8,
         "conserve": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# the most work a drawn case may cost, in pair products of the FP32 mode sum (about the largest listed case)
_COST = {"fp32": 1.0, "fp32x2": 12.0, "fp64": 60.0}
_MOST = 6e9


def _pairs(dim, N):
    """Unordered pairs (l, m) with l + m = k over the half spectrum k_1 >= 0."""
    h = N // 2 - 1
    rows = sum(k1 // 2 - (k1 - h) + 1 for k1 in range(h + 1))
    inner = sum(2 * h + 1 - abs(k) for k in range(-h, h + 1))
    return rows * inner ** (dim - 1)


def draw(rng):
    kind = rng.choice(["collide", "collide", "collide", "host", "group", "relax", "transport", "transport", "step"])
    precision = rng.choice(["fp32", "fp32", "fp32", "fp32x2", "fp64"])
    if kind in ("collide", "host", "relax"):
        dim = rng.choice([2, 2, 2, 3])
        N = rng.choice([12, 16, 20, 24, 28, 30, 32, 32, 40, 48, 64]) if dim == 2 else rng.choice([8, 12, 16])
        dirs = rng.choice([0, 0, 4, 8]) if dim == 2 and N in (16, 24, 32, 48) else 0
        if precision == "fp32x2" and (dirs or N > 48):
            precision = "fp32"
        per = _pairs(dim, N) * _COST[precision] * (20 if N > 48 else 1) * (2 if kind == "relax" else 1)
        most = int(max(40, min(65536, _MOST / per, 2 ** 26 / N ** dim)))
        c = {"kind": kind, "dim": dim, "N": N, "L": rng.choice([8.0, 10.0]), "dirs": dirs,
             "gamma": 0.0 if dirs else rng.choice([0.0, 1.0]), "conserve": rng.random() < 0.3, "precision": precision,
             "cells": _log_int(rng, 20, most), "input": rng.choice(["bi", "noisy", "shifted"])}
        if kind == "relax":
            c.update(scheme=rng.choice(["ars222", "bpr343", "euler"]), model=rng.choice(["boltzmann", "boltzmann", "bgk"]),
                     eps=rng.choice([5e-3, 0.05, 1.0]), dt=1e-3)
        return c
    if kind == "group":
        parts = []
        for _ in range(rng.randint(3, 8)):
            dim = rng.choice([2, 2, 2, 2, 3])
            N = rng.choice([16, 24, 32, 48]) if dim == 2 else 16
            most = max(60, min(20000, _MOST / 10 / (_pairs(dim, N) * _COST[precision])))
            parts.append("%d:%d:%d" % (dim, N, _log_int(rng, 50, most)))
        return {"kind": "group", "precision": precision, "instances": " ".join(parts)}
    precision = "fp32" if precision == "fp32x2" else precision
    c = {"kind": kind, "order": rng.choice([2, 2, 3]), "precision": precision, "L": 10.0}
    if rng.random() < 0.6:
        c.update(mesh="sod", size=_log_int(rng, 12, 100 if precision == "fp32" else 60), N=rng.choice([16, 24, 32, 32]))
    else:
        c.update(mesh="voronoi", size=rng.choice([300, 678, 1200, 2603]), N=rng.choice([16, 30, 32]))
    if kind == "step":
        c.update(scheme=rng.choice(["ars222", "bpr343", "euler"]), model=rng.choice(["boltzmann", "bgk"]),
                 gamma=rng.choice([0.0, 1.0]), dirs=0, eps=rng.choice([5e-3, 0.05]), conserve=rng.random() < 0.5)
        if precision == "fp64" and c["mesh"] == "sod":
            c["size"] = min(c["size"], 40)
    return c


# ---- inputs -----------------------------------------------------------------------------------------------------


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _nodes(N, L):
    return -L + (2.0 * L / N) * torch.arange(N, device="cuda", dtype=torch.float64)


def _gaussian(dim, N, L, rho, u, theta):
    """rho (2 pi theta)^(-d/2) exp(-|v - u|^2 / (2 theta)) on the grid, (cells, N^d)."""
    v = _nodes(N, L)
    out = (rho / (2 * math.pi * theta) ** (dim / 2)).reshape(-1, *([1] * dim))
    for i in range(dim):
        shape = [-1] + [1] * dim
        shape[i + 1] = N
        out = out * torch.exp(-(v[None, :] - u[:, i:i + 1]) ** 2 / (2 * theta[:, None])).reshape(shape)
    return out.reshape(len(rho), N ** dim)


def _cells(dim, N, L, cells, kind, g):
    """Two Gaussians per cell: "bi" with drifts in [-1, 1]^d, "noisy" the same with 5 % point noise, "shifted" drifting
    at Mach 0 to 3 (sound speed sqrt(2 theta))."""
    f = 0.0
    for _ in range(2):
        rho, th = _uniform(g, 0.5, 2.0, cells), _uniform(g, 0.5, 1.5, cells)
        if kind == "shifted":
            d = torch.randn((cells, dim), generator=g, device="cuda", dtype=torch.float64)
            u = d / d.norm(dim=1, keepdim=True) * (_uniform(g, 0.0, 3.0, cells) * torch.sqrt(2 * th))[:, None]
        else:
            u = _uniform(g, -1.0, 1.0, cells, dim)
        f = f + _gaussian(dim, N, L, rho, u, th)
    if kind == "noisy":
        f = f * (1.0 + 0.05 * _uniform(g, -1.0, 1.0, *f.shape))
    return f


def _instances(case):
    return [tuple(int(x) for x in p.split(":")) for p in case["instances"].split()]


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 31))
    if case["kind"] == "group":
        return [_cells(d, N, 10.0, n, "bi", g).to(_dtype(case)) for d, N, n in _instances(case)]
    if "mesh" not in case:
        f = _cells(case["dim"], case["N"], case["L"], case["cells"], case["input"], g).to(_dtype(case))
        return f.cpu().pin_memory() if case["kind"] == "host" else f
    m = _geometry(case["mesh"], case["size"])
    x, y = (torch.from_numpy(m["bary"][:, i].copy()).cuda() for i in range(2))
    n = len(x)
    if case["mesh"] == "voronoi":            # the isentropic vortex, a little perturbed
        rho, T = m["vortex"]
        rho, th = torch.from_numpy(rho).cuda(), torch.from_numpy(T).cuda()
        u = 1.0 + _uniform(g, -0.2, 0.2, n, 2)
    else:                                    # the explosion problem's two states, a little perturbed
        rho, th = torch.where(x < 0.5, 1.0, 0.125).double(), torch.where(x < 0.5, 1.0, 0.8).double()
        u = _uniform(g, -0.1, 0.1, n, 2)
    rho, th = rho * _uniform(g, 0.95, 1.05, n), th * _uniform(g, 0.95, 1.05, n)
    return _gaussian(2, case["N"], case["L"], rho, u, th).to(_dtype(case))


# ---- the handles a program keeps, and the pass ------------------------------------------------------------------


@functools.lru_cache(maxsize=None)
def _grid(dim, N, L):
    return bz.Grid(dim, N, L)


@functools.lru_cache(maxsize=None)
def _modes(dim, N, L, gamma, dirs):
    g = _grid(dim, N, L)
    return bz.FastModes(g, dirs) if dirs else bz.Modes(g, gamma)


@functools.lru_cache(maxsize=None)
def _mesh(mesh, size, order):
    pts, cells, period = _polygons(mesh, size)
    return bz.Mesh(pts, cells, order=order, periodic=period)


def _dt(case):
    if "dt" in case:
        return case["dt"]
    return 0.2 * math.sqrt(float(_geometry(case["mesh"], case["size"])["area"].mean())) / (math.sqrt(2.0) * case["L"])


def prepare(case, seed):
    s = dict(case=case, f=_inputs(case, seed))
    if case["kind"] == "group":
        s["entries"] = [(_modes(d, N, 10.0, 1.0, 0), f, torch.empty_like(f))
                        for (d, N, _), f in zip(_instances(case), s["f"])]
        return s
    s["out"] = torch.empty_like(s["f"], pin_memory=case["kind"] == "host")
    if case["kind"] != "transport":
        s["modes"] = _modes(case.get("dim", 2), case["N"], case["L"], case["gamma"], case["dirs"])
    else:
        s["grid"] = _grid(2, case["N"], case["L"])
    if "mesh" in case:
        s["mesh"] = _mesh(case["mesh"], case["size"], case["order"])
    if case["kind"] in ("step", "relax"):
        s["dt"] = _dt(case)
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "collide":
        return bz.collide_batch(s["modes"], s["f"], s["out"], precision=c["precision"], conserve=c["conserve"])
    if c["kind"] == "host":
        out = bz.collide_batch_host(s["modes"], s["f"], s["out"], precision=c["precision"], conserve=c["conserve"])
        torch.cuda.current_stream().synchronize()        # the host result is read once the stream has completed
        return out
    if c["kind"] == "group":
        bz.group_collide(s["entries"], precision=c["precision"])
        return [Q for _, _, Q in s["entries"]]
    if c["kind"] == "transport":
        return bz.transport_residual(s["mesh"], s["grid"], s["f"], s["out"], precision=c["precision"])
    if c["kind"] == "relax":
        return bz.imex_step(s["modes"], s["f"], s["dt"], c["eps"], f_out=s["out"], scheme=c["scheme"], model=c["model"],
                            precision=c["precision"], conserve=c["conserve"])
    return bz.imex_step_fv(s["modes"], s["mesh"], s["f"], s["dt"], c["eps"], f_out=s["out"], scheme=c["scheme"],
                           model=c["model"], precision=c["precision"], conserve=c["conserve"])


# ---- work -------------------------------------------------------------------------------------------------------

_TABLEAUX = {
    "ars222": (lambda g, d: ([[0] * 3, [g, 0, 0], [d, 1 - d, 0]], [[0] * 3, [0, g, 0], [0, 1 - g, g]]))(
        1 - 1 / math.sqrt(2), 1 - 1 / (2 * (1 - 1 / math.sqrt(2)))),
    "bpr343": ([[0] * 5, [1, 0, 0, 0, 0], [4 / 9, 2 / 9, 0, 0, 0], [.25, 0, .75, 0, 0], [.25, 0, .75, 0, 0]],
               [[0] * 5, [.5, .5, 0, 0, 0], [5 / 18, -1 / 9, .5, 0, 0], [.5, 0, 0, .5, 0], [.25, 0, .75, -.5, .5]]),
    "euler": ([[0, 0], [1, 0]], [[0, 0], [0, 1]]),
}


def _collide_flops(dim, N, dirs):
    """Per cell: the mode sum (a complex product and its share of the weight, nine operations a pair; or dirs / 2 + 1
    products by padded FFTs, five n log2 n a transform) and the two transforms of f and Q."""
    fft = 2 * 2.5 * N ** dim * math.log2(N ** dim)
    if dirs:
        h, P = N // 2 - 1, 3 * (N // 2)
        one = 5 * P * math.log2(P)
        return fft + (dirs // 2 + 1) * (2 * h + 1 + P) * one + (P + h + 1) * one
    return fft + 9 * _pairs(dim, N)


def work(case):
    size = 8 if case["precision"] == "fp64" else 4
    if case["kind"] == "group":
        inst = _instances(case)
        return {"bytes": sum(2 * size * n * N ** d for d, N, n in inst),
                "flops": sum(n * _collide_flops(d, N, 0) for d, N, n in inst)}
    dim, nv = case.get("dim", 2), case["N"] ** case.get("dim", 2)
    n = case["cells"] if "cells" in case else len(_polygons(case["mesh"], case["size"])[1])
    flops = 0.0
    if case["kind"] in ("collide", "host"):
        flops = n * _collide_flops(dim, case["N"], case["dirs"])
    else:
        residuals = 1
        if case["kind"] != "transport":
            At, _ = _TABLEAUX[case["scheme"]]
            used = sum(any(row[q] for row in At) for q in range(len(At)))
            residuals = used if case["kind"] == "step" else 0
            flops = n * nv * len(At) * 40.0
            if case["model"] == "boltzmann":
                flops += used * n * _collide_flops(dim, case["N"], case["dirs"])
        if residuals:
            flops += residuals * n * nv * (120.0 if case["order"] == 2 else 400.0)
    return {"bytes": 2 * size * n * nv, "flops": flops}


# ---- the same results in 64 bits --------------------------------------------------------------------------------

_RADIUS = 2.0 * (2.0 / (3.0 + math.sqrt(2.0))) * math.pi      # |q| <= 2 lambda pi


def _half_modes(dim, N, f):
    """f-hat over K_h, modes first and cells last (complex128), from f (cells, N^d)."""
    h = N // 2 - 1
    k = torch.arange(-h, h + 1, device="cuda", dtype=torch.float64)
    u = -math.pi + (2 * math.pi / N) * torch.arange(N, device="cuda", dtype=torch.float64)
    E = torch.exp(-1j * k[:, None] * u[None, :]) / N
    x = f.reshape(-1, *([N] * dim)).to(torch.complex128)
    for _ in range(dim):                      # transforms the first velocity axis and puts its modes last
        x = torch.tensordot(x, E, dims=([1], [1]))
    return x.movedim(0, -1).contiguous()


def _from_modes(dim, N, Qh, scale):
    """scale Re sum_k Q-hat_k e^{ik.u} on the grid, (cells, N^d), from all modes of K_h (modes first)."""
    h = N // 2 - 1
    k = torch.arange(-h, h + 1, device="cuda", dtype=torch.float64)
    u = -math.pi + (2 * math.pi / N) * torch.arange(N, device="cuda", dtype=torch.float64)
    E = torch.exp(1j * k[:, None] * u[None, :])
    x = Qh.movedim(-1, 0)
    for _ in range(dim):
        x = torch.tensordot(x, E, dims=([1], [0]))
    return scale * x.real.reshape(x.shape[0], N ** dim)


@functools.lru_cache(maxsize=2)
def _weights(dim, N, gamma):
    """beta-hat(l, k - l) through F(|l + m|^2, |l - m|^2) by Gauss-Legendre quadrature over |q|."""
    h = N // 2 - 1
    b0 = 1 / (2 * math.pi) if dim == 2 else 1 / (4 * math.pi)
    x, w = np.polynomial.legendre.leggauss(max(64, int(1.2 * 1.5 * _RADIUS * h * math.sqrt(dim)) + 60))
    rho, w = torch.from_numpy(0.5 * _RADIUS * (x + 1)).cuda(), torch.from_numpy(0.5 * _RADIUS * w).cuda()
    n2 = torch.arange(dim * 4 * h * h + 1, device="cuda", dtype=torch.float64)
    arg = 0.5 * torch.sqrt(n2)[:, None] * rho[None, :]
    if dim == 2:                              # J0(x) = the mean of cos(x sin t): the trapezoidal rule is exact here
        t = [math.pi * (i + 0.5) / 256 for i in range(256)]
        rad = sum(torch.cos(arg * math.sin(x)) for x in t) / len(t)
    else:
        rad = torch.sinc(arg / math.pi)
    c = (2 * math.pi if dim == 2 else 4 * math.pi) ** 2 * b0
    return c * (rad[: dim * h * h + 1] * (w * rho ** (gamma + dim - 1))) @ rad.T


def _modesum(dim, N, gamma, fh):
    """Q-hat_k = sum over l + m = k of (B(l, m) - B(m, m)) f-hat_l f-hat_m over K_h, k_1 >= 0 completed by symmetry."""
    h, M = N // 2 - 1, N - 1
    F = _weights(dim, N, gamma)
    r = torch.arange(-h, h + 1, device="cuda")
    k = torch.stack(torch.meshgrid(*([r[h:]] + [r] * (dim - 1)), indexing="ij"), -1)      # (h + 1, M, .., dim)
    k2 = (k * k).sum(-1)
    Q = torch.zeros((h + 1,) + (M,) * (dim - 1) + fh.shape[-1:], device="cuda", dtype=torch.complex128)
    grids = np.stack(np.meshgrid(*[np.arange(-h, h + 1)] * dim, indexing="ij"), -1).reshape(-1, dim)
    for l in grids.tolist():
        ks, ms = [], []
        for i in range(dim):
            lo, hi = max(0 if i == 0 else -h, l[i] - h), min(h, l[i] + h)
            ks.append(slice(lo + (0 if i == 0 else h), hi + 1 + (0 if i == 0 else h)))
            ms.append(slice(lo - l[i] + h, hi - l[i] + 1 + h))
        kk = k[tuple(ks)]
        if kk.numel() == 0:
            continue
        lv = torch.tensor(l, device="cuda")
        d2 = ((2 * lv - kk) ** 2).sum(-1)
        m2 = ((kk - lv) ** 2).sum(-1)
        beta = F[k2[tuple(ks)], d2] - F[0, 4 * m2]
        x = fh[tuple(ms)] * beta.unsqueeze(-1)
        Q[tuple(ks)].addcmul_(x, fh[tuple(v + h for v in l)].expand_as(x))
    full = torch.zeros((M,) * dim + fh.shape[-1:], device="cuda", dtype=torch.complex128)
    full[h:] = Q
    full[:h] = Q[1:].flip(list(range(dim))).conj()
    return full


def _fast_modesum(N, dirs, fh):
    """The Carleman form: sum over p of (alpha_p f-hat) * (alpha'_p f-hat) minus f-hat * (B(m, m) f-hat), by FFTs."""
    h, M, P = N // 2 - 1, N - 1, 2 * N
    k = torch.arange(-h, h + 1, device="cuda", dtype=torch.float64)
    phi = lambda x: 2 * _RADIUS * torch.sinc(_RADIUS * x / math.pi)  # noqa: E731
    f = fh.movedim(-1, 0)
    back = lambda a: torch.fft.ifft2(a * f, s=(P, P), norm="forward")  # noqa: E731
    acc, loss = 0.0, 0.0
    for p in range(dirs):
        t = math.pi * p / dirs
        e = (math.cos(t) * k[:, None] + math.sin(t) * k[None, :], -math.sin(t) * k[:, None] + math.cos(t) * k[None, :])
        a, b = phi(e[0]) / dirs, phi(e[1])                       # 2 b0 pi / dirs with b0 = 1 / (2 pi)
        acc = acc + back(a) * back(b)
        loss = loss + a * b
    acc = acc - back(torch.ones_like(loss)) * back(loss)
    return torch.fft.fft2(acc, norm="forward")[:, h:h + M, h:h + M].movedim(0, -1)


def _invariants(dim, N, L):
    v = torch.stack([x.reshape(-1) for x in torch.meshgrid(*[_nodes(N, L)] * dim, indexing="ij")])
    return torch.cat([torch.ones_like(v[:1]), v, (v * v).sum(0, keepdim=True)])


def _collide(dim, N, L, gamma, dirs, conserve, f):
    out = torch.empty_like(f)
    step = max(1, 2 ** 22 // N ** dim)
    for i in range(0, len(f), step):
        fh = _half_modes(dim, N, f[i:i + step])
        Qh = _fast_modesum(N, dirs, fh) if dirs else _modesum(dim, N, gamma, fh)
        out[i:i + step] = _from_modes(dim, N, Qh, (L / math.pi) ** (dim + gamma))
    if conserve:
        C = _invariants(dim, N, L)
        out -= torch.linalg.solve(C @ C.T, C @ out.T).T @ C
    return out


def _maxwellian(dim, N, L, f):
    C, w = _invariants(dim, N, L), (2 * L / N) ** dim
    m = w * f @ C.T
    rho, u = m[:, 0], m[:, 1:dim + 1] / m[:, :1]
    theta = (m[:, dim + 1] / rho - (u * u).sum(1)) / dim
    return rho, _gaussian(dim, N, L, rho, u, theta)


def _imex(case, f, transport):
    At, A = _TABLEAUX[case["scheme"]]
    dim, N, L, eps, dt = case.get("dim", 2), case["N"], case["L"], case["eps"], _dt(case)
    X, P = [], []
    for l in range(len(At)):
        R = f.clone()
        for q in range(l):
            if At[l][q]:
                R += dt * At[l][q] * X[q]
            if A[l][q]:
                R += (dt * A[l][q] / eps) * P[q]
        rho, M = _maxwellian(dim, N, L, R)
        c = (dt * A[l][l] / eps * rho)[:, None]
        F = (R + c * M) / (1 + c)
        P.append(rho[:, None] * (M - F))
        x = None
        if any(row[l] for row in At):
            x = -transport(F) if transport else torch.zeros_like(F)
            if case["model"] == "boltzmann":
                x += (_collide(dim, N, L, case["gamma"], case["dirs"], case["conserve"], F) - P[l]) / eps
        X.append(x)
    return F


def exact(case, seed):
    f = _inputs(case, seed)
    if case["kind"] == "group":
        return [_collide(d, N, 10.0, 1.0, 0, False, x.double()) for (d, N, _), x in zip(_instances(case), f)]
    f = f.cuda().double()
    transport = None
    if "mesh" in case:
        rec = _reconstruction(case["mesh"], case["size"], case["order"])
        transport = lambda x: _residual(rec, case["N"], case["L"], x)  # noqa: E731
    if case["kind"] == "transport":
        return transport(f)
    if case["kind"] in ("step", "relax"):
        return _imex(case, f, transport)
    return _collide(case["dim"], case["N"], case["L"], case["gamma"], case["dirs"], case["conserve"], f)


# ---- meshes and the 64-bit transport residual -------------------------------------------------------------------


@functools.lru_cache(maxsize=None)
def _polygons(mesh, size):
    """(vertices, counter-clockwise cells, periods): the explosion problem's triangles or the vortex study's polygons."""
    if mesh == "voronoi":
        pts, cells = workloads.periodic_voronoi(size)
        period = (10.0, 10.0)
    else:
        pts, cells = workloads.sod_triangulation(size)
        period = None
    out = []
    for c in cells:
        x, y = (pts[list(c)] - pts[c[0]]).T
        ccw = (x * np.roll(y, -1) - np.roll(x, -1) * y).sum() > 0
        out.append([int(v) for v in (c if ccw else c[::-1])])
    return pts, out, period


@functools.lru_cache(maxsize=None)
def _geometry(mesh, size):
    pts, cells, _ = _polygons(mesh, size)
    n = len(cells)
    area, bary, h = np.zeros(n), np.zeros((n, 2)), np.zeros(n)
    for i, c in enumerate(cells):
        p = pts[c] - pts[c[0]]
        x, y = p.T
        xn, yn = np.roll(x, -1), np.roll(y, -1)
        cr = x * yn - xn * y
        area[i] = 0.5 * cr.sum()
        bary[i] = pts[c[0]] + np.array([((x + xn) * cr).sum(), ((y + yn) * cr).sum()]) / (6 * area[i])
        h[i] = np.sqrt(((pts[c] - bary[i]) ** 2).sum(1)).max()
    g = {"area": area, "bary": bary, "h": h}
    if mesh == "voronoi":
        dx = bary % 10.0 - 5.0
        dT = -25.0 / (16.0 * math.pi ** 2) * np.exp(1.0 - (dx ** 2).sum(1))
        g["vortex"] = (1.0 + dT, 1.0 + dT)
    return g


def _means(p, xb, h):
    """Means over the polygon p of (xi, eta, xi^2, xi eta, eta^2), xi and eta from xb in units of h (a fan of triangles,
    each by its edge midpoints, exact for quadratics)."""
    q = (p - xb) / h
    a, b, c = q[:1].repeat(len(q) - 2, 0), q[1:-1], q[2:]
    w = 0.5 * ((b - a)[:, 0] * (c - a)[:, 1] - (c - a)[:, 0] * (b - a)[:, 1])
    m = np.concatenate([0.5 * (a + b), 0.5 * (b + c), 0.5 * (c + a)])
    w = np.tile(w, 3) / (3 * w.sum())
    x, y = m.T
    return np.array([(w * t).sum() for t in (x, y, x * x, x * y, y * y)])


@functools.lru_cache(maxsize=2)
def _reconstruction(mesh, size, order):
    """Faces, stencils and least-squares matrices of the CWENO reconstruction (degree order - 1) as device tensors."""
    pts, cells, period = _polygons(mesh, size)
    geo = _geometry(mesh, size)
    bary, hs, n = geo["bary"], geo["h"], len(cells)
    per = np.array(period if period else (0.0, 0.0))
    lattice = (lambda s: tuple(np.round(s / per) * per)) if period else (lambda s: (0.0, 0.0))
    if period:                               # one index for all periodic images of a vertex: clusters of x and of y
        cls = 0
        for x, p in zip((pts % per).T, per):
            x = np.where(x > p - 1e-7, x - p, x)
            by = np.argsort(x)
            rank = np.empty(len(x), np.int64)
            rank[by] = np.cumsum(np.diff(x[by], prepend=x[by[0]]) > 1e-7)
            cls = cls * len(x) + rank
        cls = np.unique(cls, return_inverse=True)[1]
    else:
        cls = np.arange(len(pts))
    owner, at = {}, {}
    for i, c in enumerate(cells):
        for q, a in enumerate(c):
            owner[cls[a], cls[c[(q + 1) % len(c)]]] = (i, c[(q + 1) % len(c)])
            at.setdefault(int(cls[a]), []).append((i, a))
    near = []                                # cells sharing a vertex, with their translations
    for i, c in enumerate(cells):
        s = {(j, *lattice(pts[v] - pts[w])) for v in c for j, w in at[int(cls[v])]}
        s.discard((i, 0.0, 0.0))
        near.append(s)
    K, W = (11 if order == 3 else 5), max(len(c) for c in cells)
    st = np.zeros((n, K), np.int64)
    nb, geom, shift = np.full((n, W), -1, np.int64), np.zeros((n, W, 3)), np.zeros((n, W, 2))
    ends = np.zeros((n, W, 2, 2))
    sec = np.zeros((n, W, 2, 2))             # per sector: the gradient (in units of 1 / h) from two differences
    sid, nsec = np.zeros((n, W, 2), np.int64), np.zeros(n)
    where, rel = bary.tolist(), np.zeros((n, K, 2))
    for i, c in enumerate(cells):
        x, y = where[i]
        cand = {(k, sx + tx, sy + ty) for j, sx, sy in near[i] for k, tx, ty in near[j]} | near[i]
        cand.discard((i, 0.0, 0.0))
        cand = sorted((math.hypot(where[j][0] + sx - x, where[j][1] + sy - y), j, sx, sy) for j, sx, sy in cand)[:K]
        st[i], rel[i] = [t[1] for t in cand], [(where[j][0] + sx - x, where[j][1] + sy - y) for _, j, sx, sy in cand]
    second = np.array([_means(pts[c], bary[i], 1.0) for i, c in enumerate(cells)])[:, 2:]
    mu = second / hs[:, None] ** 2           # means of xi^2, xi eta, eta^2 over the cell itself
    rel /= hs[:, None, None]
    a = rel
    if order == 3:                           # the basis' means over the stencil's cells
        e = np.stack([rel[..., 0] ** 2, rel[..., 0] * rel[..., 1], rel[..., 1] ** 2], -1)
        a = np.concatenate([rel, e + second[st] / hs[:, None, None] ** 2 - mu[:, None]], -1)
    opt = np.linalg.solve(a.transpose(0, 2, 1) @ a, a.transpose(0, 2, 1))
    for i, c in enumerate(cells):
        h = hs[i]
        off = []
        for q, a0 in enumerate(c):
            a1 = c[(q + 1) % len(c)]
            d = pts[a1] - pts[a0]
            geom[i, q] = (math.hypot(*d), d[1] / math.hypot(*d), -d[0] / math.hypot(*d))
            ends[i, q] = pts[a0], pts[a1]
            o = owner.get((cls[a1], cls[a0]))
            if o is not None:                # o[1] is the neighbour's copy of a0
                nb[i, q] = o[0]
                shift[i, q] = lattice(pts[a0] - pts[o[1]])
            off.append((bary[nb[i, q]] + shift[i, q] - bary[i]) / h)
        for q in range(len(c)):
            q2 = (q + 1) % len(c)
            if nb[i, q] < 0 or nb[i, q2] < 0:
                continue
            a = np.array([off[q], off[q2]])
            if abs(a[0, 0] * a[1, 1] - a[0, 1] * a[1, 0]) <= 1e-12 * np.abs(a).max() ** 2:
                continue
            k = int(nsec[i])
            sec[i, k], sid[i, k] = a, (nb[i, q], nb[i, q2])
            nsec[i] += 1
    for q in range(W):
        sec[nsec > q, q] = np.linalg.inv(sec[nsec > q, q])
    r = dict(st=st, opt=opt, nb=nb, geom=geom, shift=shift, ends=ends, mu=mu, sec=sec, sid=sid, nsec=nsec, bary=bary,
             h=hs, area=geo["area"])
    r = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in r.items()}
    r["order"] = order
    return r


def _residual(r, N, L, f):
    """(1 / |P|) sum over the faces of |e| times the upwind (Rusanov) flux of the reconstructed face values."""
    n, nv = f.shape
    quad, W = r["order"] == 3, r["nb"].shape[1]
    B = 5 if quad else 2
    C = torch.zeros((n, B, nv), device="cuda", dtype=torch.float64)
    size = max(1, 2 ** 24 // (12 * nv))
    mu = r["mu"][:, :, None]
    for i in range(0, n, size):
        s = slice(i, i + size)
        f0, m = f[s][:, None], mu[s]
        opt = torch.bmm(r["opt"][s], f[r["st"][s]] - f0)
        lam = torch.where(r["nsec"][s] > 0, 0.25 / r["nsec"][s].clamp(min=1), 0.0)[:, None, None]
        polys, lams = [], []
        for q in range(W):
            on = (r["nsec"][s] > q)[:, None, None]
            g = torch.zeros_like(opt)
            g[:, :2] = torch.bmm(r["sec"][s][:, q], f[r["sid"][s][:, q]] - f0)
            polys.append(g * on)
            lams.append(lam * on)
        lam0 = 1.0 - sum(lams)
        polys.insert(0, (opt - sum(a * b for a, b in zip(lams, polys))) / lam0)
        lams.insert(0, lam0)
        tot, acc = 0.0, 0.0
        for a, p in zip(lams, polys):
            sig = p[:, 0] ** 2 + p[:, 1] ** 2
            if quad:
                c3, c4, c5 = p[:, 2], p[:, 3], p[:, 4]
                m2, m11, m02 = m[:, 0], m[:, 1], m[:, 2]
                sig = sig + 4 * c3 * c3 * m2 + 4 * c3 * c4 * m11 + c4 * c4 * (m02 + m2) + 4 * c4 * c5 * m11 \
                    + 4 * c5 * c5 * m02 + 4 * c3 * c3 + c4 * c4 + 4 * c5 * c5
            w = a / (sig[:, None] + 1e-14) ** 4
            tot, acc = tot + w, acc + w * p
        C[s] = acc / tot
    v = _nodes(N, L)
    v1, v2 = v.repeat_interleave(N)[None], v.repeat(N)[None]
    points = (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)) if quad else (0.5,)

    def value(cell, x):
        xi = (x - r["bary"][cell]) / r["h"][cell][:, None]
        phi = [xi[:, 0], xi[:, 1]]
        if quad:
            m = r["mu"][cell]
            phi += [xi[:, 0] ** 2 - m[:, 0], xi[:, 0] * xi[:, 1] - m[:, 1], xi[:, 1] ** 2 - m[:, 2]]
        return f[cell] + torch.bmm(torch.stack(phi, 1)[:, None], C[cell])[:, 0]

    out = torch.zeros_like(f)
    for i in range(0, n, size):
        me = torch.arange(i, min(n, i + size), device="cuda")
        acc = 0.0
        for q in range(W):
            ln, nx, ny = (r["geom"][me, q, k][:, None] for k in range(3))
            vn = v1 * nx + v2 * ny
            j = r["nb"][me, q]
            for t in points:
                x = r["ends"][me, q, 0] + t * (r["ends"][me, q, 1] - r["ends"][me, q, 0])
                fl = value(me, x)
                fr = torch.where((j >= 0)[:, None], value(j.clamp(min=0), x - r["shift"][me, q]), fl)
                acc = acc + ln / len(points) * (0.5 * vn * (fl + fr) - 0.5 * vn.abs() * (fr - fl))
        out[i:i + size] = acc / r["area"][me][:, None]
    return out
