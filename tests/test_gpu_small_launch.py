"""Launch rules of the mode sums: small batches (two outputs per thread, tiles
split over CTAs, programmatic launches) and split FP64 / FP32X2 tiles give every
cell the bits it has in a large batch; the 8-cell form on 64^2 and 16^3 against
the oracle."""
import pytest

from paper_2103_14890_gb300 import workloads
from gpu_util import as_input, bz_module, check_fp32_cells, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bz():
    return bz_module()


@pytest.mark.parametrize("dim,N,precision", [(2, 16, "fp32"), (2, 30, "fp32"), (2, 32, "fp32"), (2, 48, "fp32"),
                                             (2, 64, "fp32"), (3, 16, "fp32"), (2, 32, "fp64"), (2, 6, "fp64"),
                                             (2, 48, "fp32x2"), (3, 16, "fp32x2")])
def test_batches_agree_bit_for_bit(bz, dim, N, precision):
    import torch
    n = 4900 if dim == 2 and N <= 32 and precision == "fp32" else 700
    f = to_dev(workloads.bi_maxwellian(n, dim, N, 10.0, seed=N), precision)
    m = bz.Modes(bz.Grid(dim, N, 10.0), 1.0)
    want = bz.collide_batch(m, f, precision=precision)
    for k in (1, 17, 64, 303, 699):
        for _ in range(2):               # back to back: a launch starts while the one before it ends
            got = bz.collide_batch(m, f[:k].contiguous(), precision=precision)
        assert torch.equal(got, want[:k]), k
    bz.check()


@pytest.mark.parametrize("dim,N,n", [(2, 64, 1), (2, 64, 9), (2, 62, 8), (3, 16, 33)])
def test_eight_cell_form(bz, dim, N, n):
    import oracle
    f = workloads.bi_maxwellian(n, dim, N, 10.0, seed=7, noise=0.05)
    fin = as_input(f, "fp32")
    k = oracle.Kernel(dim, N, 10.0, 1.0)
    got = bz.collide_batch(bz.Modes(bz.Grid(dim, N, 10.0), 1.0), to_dev(f, "fp32"), precision="fp32", conserve=True)
    bz.check()
    want = k.collide(fin, conserve=True)
    got = got.double().cpu().numpy()
    check_fp32_cells(k, fin, got, want, what="%dd N=%d" % (dim, N))


@pytest.mark.parametrize("dim,N,precision,sizes", [
    (2, 24, "fp32", (500, 1949, 7000)), (2, 32, "fp32", (2500, 5000, 9001)), (2, 48, "fp32", (1300, 3000, 6001)),
    (2, 64, "fp32", (100, 700, 1501)), (3, 16, "fp32", (100, 700, 1401)), (2, 32, "fp64", (300, 2000)),
    (2, 48, "fp32x2", (301, 1000))])
def test_shared_tail_tiles(bz, dim, N, precision, sizes):
    """Batches whose last tiles are shared by 2 to 8 CTAs: the bits of a batch that ends elsewhere."""
    import torch
    f = to_dev(workloads.bi_maxwellian(max(sizes), dim, N, 10.0, seed=N + 1), precision)
    m = bz.Modes(bz.Grid(dim, N, 10.0), 1.0)
    want = torch.cat([bz.collide_batch(m, part.contiguous(), precision=precision) for part in f.split(487)])
    for n in sizes:
        assert torch.equal(bz.collide_batch(m, f[:n].contiguous(), precision=precision), want[:n]), n
    bz.check()
