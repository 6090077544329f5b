"""The FP32 transport passes on triangle meshes at sizes where a block takes many
cells in turn (the value passes of degree 1, the staged pass of degree 2) and at
the edges of their dispatch: against the FP64 passes on the same data, cell by
cell, and the two-sided steps against steps of tiny dt in FP64."""
import numpy as np
import pytest

from paper_2103_14890_gb300 import workloads
from gpu_util import bz_module

pytestmark = pytest.mark.gpu
U32 = 2.0 ** -24


@pytest.fixture(scope="module")
def bz():
    return bz_module()


def _mesh(size):
    """A triangulation of about 2 size^2 cells, and per cell perimeter / area."""
    pts, tri = workloads.sod_triangulation(size)
    a, b, c = (pts[tri[:, k]] for k in range(3))
    area = 0.5 * np.abs((b - a)[:, 0] * (c - a)[:, 1] - (b - a)[:, 1] * (c - a)[:, 0])
    per = sum(np.hypot(*(x - y).T) for x, y in ((a, b), (b, c), (c, a)))
    return pts, tri, per / area


def _check(got, want, per_area, L, fmax, extra=0.0):
    """64 roundings of the magnitudes summed: a cell's faces times both sides' states, each at most 16 times the
    largest average (the reconstruction's rows on a jittered lattice).  Slivers, where these grow, are left out."""
    keep = per_area < 50.0 * np.median(per_area)
    bound = 64 * U32 * per_area * 1.25 * L * 2 * 17 * fmax + extra
    err = np.abs(got - want).max(1)
    assert keep.mean() > 0.98 and np.isfinite(got[keep]).all()
    assert (err[keep] <= bound[keep]).all(), float((err / bound)[keep].max())
    # rounding is no systematic error: a wrong row or table entry would show as one of order one
    rms = np.sqrt(((got - want)[keep] ** 2).mean() / (want[keep] ** 2).mean())
    assert rms < 1e-4, rms


@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("size,N", [(70, 12), (70, 16), (70, 20), (70, 24), (70, 28), (70, 32), (70, 36), (20, 24), (20, 32),
                                    (100, 32)])
def test_many_cells_per_block(bz, size, N, order):
    import torch
    pts, tri, per_area = _mesh(size)
    L = 6.0
    f = 1.0 + torch.rand((len(tri), N * N), generator=torch.Generator(device="cuda").manual_seed(N), device="cuda")
    m, g = bz.Mesh(pts, tri, order=order), bz.Grid(2, N, L)
    got = bz.transport_residual(m, g, f, precision="fp32")
    want = bz.transport_residual(m, g, f.double(), precision="fp64")
    bz.check()
    _check(got.double().cpu().numpy(), want.cpu().numpy(), per_area, L, 2.0)


@pytest.mark.parametrize("size,N", [(70, 24), (70, 32), (70, 28), (40, 16)])
def test_two_sided_steps(bz, size, N):
    """Order 3 with thin cells: one Euler step without collisions (eps = 1e30) is f - dt L(f), so (f - f_out) / dt
    against L in FP64; dt L is below f but for slivers, and f_out's roundings are four of f over dt."""
    import torch
    pts, tri, per_area = _mesh(size)
    L, dt = 6.0, 2.0 ** -13
    f = 1.0 + torch.rand((len(tri), N * N), generator=torch.Generator(device="cuda").manual_seed(N), device="cuda")
    m, modes = bz.Mesh(pts, tri, order=3), bz.Modes(bz.Grid(2, N, L), 0.0)
    out = bz.imex_step_fv(modes, m, f, dt, 1e30, scheme="euler", model="bgk", precision="fp32")
    want = bz.transport_residual(m, bz.Grid(2, N, L), f.double(), precision="fp64")
    bz.check()
    got = (f.double() - out.double()) / dt
    _check(got.cpu().numpy(), want.cpu().numpy(), per_area, L, 2.0, 4 * U32 * 2.0 / dt)


def test_two_sided_polygon_steps(bz):
    """The same on quadrilaterals with thin cells, N divisible by four and not."""
    import torch
    x = np.linspace(0.0, 1.0, 31)
    x[16] = x[15] + (x[16] - x[15]) / 300
    X, Y = np.meshgrid(x, np.linspace(0.0, 1.0, 31), indexing="ij")
    i = np.arange(X.size).reshape(X.shape)
    cells = np.stack([i[:-1, :-1], i[1:, :-1], i[1:, 1:], i[:-1, 1:]], -1).reshape(-1, 4)
    pts = np.stack([X.ravel(), Y.ravel()], 1)
    w, h = np.ptp(pts[cells], axis=1).T
    L, dt = 6.0, 2.0 ** -13
    for N in (16, 32, 6):
        f = 1.0 + torch.rand((len(cells), N * N), generator=torch.Generator(device="cuda").manual_seed(N), device="cuda")
        m, modes = bz.Mesh(pts, cells, order=3), bz.Modes(bz.Grid(2, N, L), 0.0)
        out = bz.imex_step_fv(modes, m, f, dt, 1e30, scheme="euler", model="bgk", precision="fp32")
        want = bz.transport_residual(m, bz.Grid(2, N, L), f.double(), precision="fp64")
        bz.check()
        got = (f.double() - out.double()) / dt
        keep = w > 0.5 * np.median(w)
        # the thin cells' neighbours take part; the thin cells' own sums cancel by 300 more and are left out
        _check(got.cpu().numpy()[keep], want.cpu().numpy()[keep], (2 * (w + h) / (w * h))[keep], L, 2.0, 4 * U32 * 2.0 / dt)
