"""Kernels launched while the one before them ends read that one's results, not
what the scratch held before: calls on changing inputs, back to back, against
the same calls one at a time."""
import pytest

from paper_2103_14890_gb300 import workloads
from gpu_util import bz_module

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bz():
    return bz_module()


def _alternate(call, inputs):
    """call(f, out) for every input on its own, then 40 rounds of all of them without a wait in between."""
    import torch
    want = []
    for f in inputs:
        want.append(call(f, torch.empty_like(f)))
        torch.cuda.synchronize()
    outs = [[torch.full_like(f, float("nan")) for f in inputs] for _ in range(40)]
    for row in outs:
        for f, o in zip(inputs, row):
            call(f, o)
    torch.cuda.synchronize()
    for row in outs:
        for o, w in zip(row, want):
            assert torch.equal(o, w)


@pytest.mark.parametrize("precision,N", [("fp32", 8), ("fp32", 6), ("fp32", 32), ("fp64", 6), ("fp64", 16)])
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("kind", ["tri", "voronoi"])
def test_transport_back_to_back(bz, kind, order, precision, N):
    import torch
    pts, cells = workloads.sod_triangulation(20) if kind == "tri" else workloads.periodic_voronoi(100)
    mesh = bz.Mesh(pts, cells, order=order, periodic=None if kind == "tri" else (10.0, 10.0))
    grid = bz.Grid(2, N, 6.0)
    g = torch.Generator(device="cuda").manual_seed(1)
    dt = torch.float64 if precision == "fp64" else torch.float32
    inputs = [(1.0 + torch.rand((len(cells), N * N), generator=g, device="cuda", dtype=torch.float64)).to(dt) * s
              for s in (1.0, 3.0, 0.1)]
    _alternate(lambda f, o: bz.transport_residual(mesh, grid, f, o, precision=precision), inputs)


@pytest.mark.parametrize("N,n", [(16, 1), (16, 64), (24, 40), (32, 64), (48, 33)])
def test_small_batches_back_to_back(bz, N, n):
    from gpu_util import to_dev
    m = bz.Modes(bz.Grid(2, N, 8.0), 1.0)
    f = to_dev(workloads.bi_maxwellian(n, 2, N, 8.0, seed=3), "fp32")
    _alternate(lambda x, o: bz.collide_batch(m, x, o, precision="fp32"), [f, 3.0 * f, 0.1 * f])
