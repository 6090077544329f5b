"""The numbering of the faces' rows in the transport passes on unusual polygons:
edges of no length, an edge walked both ways by one cell, an edge as long as a
period.  On data linear in space every reconstruction is exact, so L = v . grad f
in every cell (transmissive boundaries and such edges included)."""
import numpy as np
import pytest

from gpu_util import bz_module, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bz():
    return bz_module()


def _lattice(n=8):
    x = np.linspace(0.0, 1.0, n + 1)
    X, Y = np.meshgrid(x, x, indexing="ij")
    rng = np.random.default_rng(4)
    X[1:-1, 1:-1] += rng.uniform(-0.2, 0.2, (n - 1, n - 1)) / n
    Y[1:-1, 1:-1] += rng.uniform(-0.2, 0.2, (n - 1, n - 1)) / n
    i = np.arange((n + 1) ** 2).reshape(n + 1, n + 1)
    return np.stack([X.ravel(), Y.ravel()], 1), np.stack([i[:-1, :-1], i[1:, :-1], i[1:, 1:], i[:-1, 1:]], -1).reshape(-1, 4)


def _repeated():
    """Every cell names its first corner twice: an edge of no length, its own reverse."""
    pts, quads = _lattice()
    return pts, [np.roll([q[0], *q], k % 5).tolist() for k, q in enumerate(quads)], None


def _slit():
    """Every second cell has a slit from a corner to its centre, walked in both directions."""
    pts, quads = _lattice()
    cells = []
    for k, q in enumerate(quads.tolist()):
        if k % 2:
            q = [q[0], len(pts), q[0]] + q[1:]
            pts = np.concatenate([pts, pts[quads[k]].mean(0, keepdims=True)])
        cells.append(q)
    return pts, cells, None


def _band():
    """Periodic in x: rows of three cells between two cells as wide as the period, whose outer edges pair with themselves."""
    y = np.linspace(0.0, 1.0, 7)
    pts = np.array([(a / 3.0, b) for b in y for a in range(4)])
    i = np.arange(28).reshape(7, 4)
    cells = [[i[0, 0], i[0, 3], *i[1, ::-1]]]
    cells += [[i[r, a], i[r, a + 1], i[r + 1, a + 1], i[r + 1, a]] for r in range(1, 5) for a in range(3)]
    cells += [[*i[5], i[6, 3], i[6, 0]]]
    return pts, [[int(v) for v in c] for c in cells], (1.0, 0.0)


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("precision,N", [("fp32", 8), ("fp32", 6), ("fp64", 6)])
@pytest.mark.parametrize("kind", ["repeated", "slit", "band"])
def test_linear_data_on_unusual_polygons(bz, kind, precision, N, order):
    Lv = 6.0
    pts, cells, per = {"repeated": _repeated, "slit": _slit, "band": _band}[kind]()
    rng = np.random.default_rng(5)
    a, b = rng.uniform(1.0, 2.0, N * N), rng.uniform(-0.4, 0.4, (2, N * N))
    if per:
        b[0] = 0.0                                     # periodic data
    f, scale = np.empty((len(cells), N * N)), np.empty(len(cells))
    for i, c in enumerate(cells):
        p = pts[c] - pts[c[0]]
        x, y = p.T
        cr = x * np.roll(y, -1) - np.roll(x, -1) * y
        xb = pts[c[0]] + ((p + np.roll(p, -1, 0)) * cr[:, None]).sum(0) / (3.0 * cr.sum())
        f[i] = a + xb @ b
        scale[i] = np.abs(np.roll(p, -1, 0) - p).sum() / (0.5 * cr.sum())
    v = -Lv + 2.0 * Lv / N * np.arange(N)
    want = np.repeat(v, N) * b[0] + np.tile(v, N) * b[1]
    mesh = bz.Mesh(pts, cells, order=order, periodic=per)
    got = bz.transport_residual(mesh, bz.Grid(2, N, Lv), to_dev(f, precision), precision=precision).double().cpu().numpy()
    bz.check()
    # 64 roundings of the magnitudes summed (as in test_gpu_transport.py): both sides' face values, each the average
    # plus a gradient whose least-squares rows, times the distance to the face, sum to at most 16 on these cells
    u = 2.0 ** -53 if precision == "fp64" else 2.0 ** -24
    bound = 64 * u * scale[:, None] * 1.25 * Lv * 2.0 * (1.0 + 2.0 * 16.0) * np.abs(f).max()
    err = np.abs(got - want)
    assert (err <= bound).all(), float((err / bound).max())


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("order", [1, 2, 3])
@pytest.mark.parametrize("precision,N", [("fp32", 8), ("fp32", 6), ("fp64", 6)])
def test_non_finite_values_stay_local(bz, precision, N, order, value):
    """A NaN or infinity at one velocity of one cell: L is not finite there, other velocities and cells two stencils
    away keep their bits."""
    import torch
    pts, quads = _lattice(12)
    mesh, grid = bz.Mesh(pts, quads.tolist(), order=order), bz.Grid(2, N, 6.0)
    f = to_dev(np.random.default_rng(6).uniform(1.0, 2.0, (len(quads), N * N)), precision)
    want = bz.transport_residual(mesh, grid, f, precision=precision)
    c, k = 6 * 12 + 6, N + 3
    f[c, k] = value
    got = bz.transport_residual(mesh, grid, f, precision=precision)
    bz.check()
    assert not torch.isfinite(got[c, k])
    other = torch.arange(N * N, device="cuda") != k
    assert torch.equal(got[:, other], want[:, other])
    i = torch.arange(len(quads), device="cuda")
    far = ((i // 12 - 6).abs() > 5) | ((i % 12 - 6).abs() > 5)
    assert far.any() and torch.equal(got[far], want[far])
