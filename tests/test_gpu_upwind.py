"""The transport passes and the IMEX stage kernel where their dispatch changes:
thin cells (two-sided sums), grids whose N is not a multiple of four, walls on
thin cells, and stage kernels on grids without a compile-time N.  Bounds as in
test_gpu_transport.py; the FP64 step within 1e-12 of the oracle."""
import numpy as np
import pytest

from paper_2103_14890_gb300 import workloads
from gpu_util import as_input, bz_module, relerr, to_dev
from test_gpu_transport import ETA32, ETA64, U32, U64, _check, _check3, _magnitude3, _walls

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bz():
    return bz_module()


@pytest.fixture(scope="module")
def fvo():
    from oracle import fv
    return fv


def _thin_mesh():
    """A structured triangulation with one lattice column squeezed to 1/400 of
    its width: thin cells inside the domain and on its boundary."""
    x = np.array([0.0, 0.2, 0.4, 0.4005, 0.6, 0.8, 0.9995, 1.0])
    X, Y = np.meshgrid(x, np.linspace(0.0, 1.0, 6), indexing="ij")
    rng = np.random.default_rng(2)
    Y[:, 1:-1] += rng.uniform(-0.03, 0.03, Y[:, 1:-1].shape)
    idx = np.arange(X.size).reshape(X.shape)
    a, b, c, d = (v.ravel() for v in (idx[:-1, :-1], idx[1:, :-1], idx[:-1, 1:], idx[1:, 1:]))
    return np.stack([X.ravel(), Y.ravel()], 1), np.concatenate([np.stack([a, b, d], 1), np.stack([a, d, c], 1)])


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("order", [2, 3])
@pytest.mark.parametrize("precision,N", [("fp32", 8), ("fp32", 6), ("fp64", 6)])
def test_thin_cells(bz, fvo, precision, N, order, walls):
    if walls and N % 4:
        pytest.skip("walls need N divisible by 4")
    pts, tri = _thin_mesh()
    om = fvo.Mesh(pts, tri)
    f = workloads.mesh_states(om.bary, N, 6.0)
    fin = as_input(f, precision)
    m = bz.Mesh(pts, tri, order=order)
    wl = None
    if walls:
        edges, params, wl = _walls(om)
        m.set_walls(np.concatenate([edges[:1], edges]), np.concatenate([params[:1] * 0.5, params]))   # an edge twice
    Lr = bz.transport_residual(m, bz.Grid(2, N, 6.0), to_dev(f, precision), precision=precision)
    bz.check()
    u, eta = (U64, ETA64) if precision == "fp64" else (U32, ETA32)
    want = fvo.transport_residual(om, fin, N, 6.0, order=order, walls=wl)
    got = Lr.double().cpu().numpy()
    if order == 2:
        _check(got, want, om, fin, N, 6.0, 2, fvo, u, eta, wl)
    else:
        _check3(got, want, om, fin, N, 6.0, fvo, u, eta, wl)


@pytest.mark.parametrize("model", ["boltzmann", "bgk"])
@pytest.mark.parametrize("dim,N,scheme", [(2, 30, "bpr343"), (2, 34, "ars222"), (3, 6, "bpr343")])
def test_stage_kernels_fp64(bz, dim, N, scheme, model):
    import oracle
    f = workloads.bi_maxwellian(3, dim, N, 8.0, seed=5)
    m = bz.Modes(bz.Grid(dim, N, 8.0), 0.0)
    got = bz.imex_step(m, to_dev(f, "fp64"), 2e-3, 5e-2, scheme=scheme, model=model, precision="fp64")
    bz.check()
    want = oracle.Kernel(dim, N, 8.0, 0.0).imex_step(f, 2e-3, 5e-2, scheme=scheme, model=model)
    assert relerr(got.cpu().numpy(), want) < 1e-12


@pytest.mark.parametrize("N", [12, 16, 20, 24, 28])
def test_value_pass_blocks(bz, fvo, N):
    """The FP32 triangle passes of degree 1 with 64, 128, 160 and 256 threads, the last warp not always full."""
    pts, tri = workloads.sod_triangulation(18, jitter=0.2)
    om = fvo.Mesh(pts, tri)
    f = workloads.mesh_states(om.bary, N, 6.0)
    fin = as_input(f, "fp32")
    Lr = bz.transport_residual(bz.Mesh(pts, tri, order=2), bz.Grid(2, N, 6.0), to_dev(f, "fp32"), precision="fp32")
    bz.check()
    _check(Lr.double().cpu().numpy(), fvo.transport_residual(om, fin, N, 6.0, order=2), om, fin, N, 6.0, 2, fvo, U32, ETA32)


@pytest.mark.parametrize("N", [12, 16, 20, 24, 28])
def test_degree2_pass_blocks(bz, fvo, N):
    """As test_value_pass_blocks for the staged pass of degree 2."""
    pts, tri = workloads.sod_triangulation(18, jitter=0.2)
    om = fvo.Mesh(pts, tri)
    f = workloads.mesh_states(om.bary, N, 6.0)
    fin = as_input(f, "fp32")
    Lr = bz.transport_residual(bz.Mesh(pts, tri, order=3), bz.Grid(2, N, 6.0), to_dev(f, "fp32"), precision="fp32")
    bz.check()
    _check3(Lr.double().cpu().numpy(), fvo.transport_residual(om, fin, N, 6.0, order=3), om, fin, N, 6.0, fvo, U32, ETA32)


@pytest.mark.parametrize("N", [8, 6])
def test_two_sided_step(bz, fvo, N):
    """A step of degree 2 on a mesh with thin cells (every face two-sided), as good as without collisions (eps = 1e30):
    f - dt L(f) of the oracle, within dt times the bound of L and four roundings of the terms."""
    pts, tri = _thin_mesh()
    om = fvo.Mesh(pts, tri)
    f = workloads.mesh_states(om.bary, N, 6.0)
    fin = as_input(f, "fp32")
    dt = 2e-5
    m = bz.Modes(bz.Grid(2, N, 6.0), 0.0)
    got = bz.imex_step_fv(m, bz.Mesh(pts, tri, order=3), to_dev(f, "fp32"), dt, 1e30, scheme="euler", model="bgk",
                          precision="fp32")
    bz.check()
    L = fvo.transport_residual(om, fin, N, 6.0, order=3)
    M = _magnitude3(om, fin, N, 6.0, fvo, None)
    bound = 64 * dt * (U32 * M + ETA32 * _magnitude3(om, np.ones_like(fin), N, 6.0, fvo, None))
    bound += 4 * U32 * (np.abs(fin) + dt * np.abs(L)) + 4 * ETA32
    err = np.abs(got.double().cpu().numpy() - (fin - dt * L))
    assert (err <= bound).all(), float((err / bound).max())
