"""FP32 stages of the BGK model in the fluid limit, on grids whose dv is no FP32
number: the stage value against FP64, point by point and in its mean momentum and
temperature (a bias in the moments would add up over the stages).

Point bound: with x the exponent, F = (R + c M) / (1 + c) carries |x| u from the
rounded exponent, 4 u from the exponential (2 ulp), one u each from the prefactor
and its product, four from c M, the sum and the quotient, and one for the
parameters: (|x| + 11) u M, u = 2^-24, and a few times the smallest subnormal."""
import numpy as np
import pytest

from paper_2103_14890_gb300 import workloads
from gpu_util import U32, as_input, bz_module, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bz():
    return bz_module()


@pytest.mark.parametrize("dim,N,L,n", [(2, 12, 5.0, 2000), (2, 20, 8.0, 2000), (2, 28, 10.0, 2000), (2, 30, 10.0, 2000),
                                       (2, 30, 8.0, 2000), (2, 40, 10.0, 500), (2, 34, 8.0, 500), (3, 10, 6.0, 500),
                                       (3, 16, 8.0, 100)])
def test_fluid_limit_stage_fp32(bz, dim, N, L, n):
    f = workloads.bi_maxwellian(n, dim, N, L, seed=N)
    fin = as_input(f, "fp32")
    dt, eps = 1e-3, 1e-8
    m = bz.Modes(bz.Grid(dim, N, L), 0.0)
    got = bz.imex_step(m, to_dev(f, "fp32"), dt, eps, scheme="euler", model="bgk", precision="fp32").double().cpu().numpy()
    bz.check()
    v = np.stack([a.ravel() for a in np.meshgrid(*[-L + 2.0 * L / N * np.arange(N)] * dim, indexing="ij")])
    w = (2.0 * L / N) ** dim

    def moments(g):
        rho = w * g.sum(1)
        u = w * (g @ v.T) / rho[:, None]
        return rho, u, (w * (g @ (v * v).sum(0)) / rho - (u * u).sum(1)) / dim

    rho, u, th = moments(fin)
    x = -((v[None] - u[:, :, None]) ** 2).sum(1) / (2.0 * th[:, None])
    pref = rho[:, None] / (2.0 * np.pi * th[:, None]) ** (dim / 2)
    M = pref * np.exp(x)
    c = (dt * rho / eps)[:, None]
    want = (fin + c * M) / (1.0 + c)
    bound = (np.abs(x) + 11.0) * U32 * want + 16.0 * 2.0 ** -149 * np.maximum(pref, 1.0)
    err = np.abs(got - want)
    assert (err <= bound).all(), float((err / bound).max())
    _, ug, tg = moments(got)
    _, uw, tw = moments(want)
    du, dth = (ug - uw).mean(0), (tg / tw - 1.0).mean()
    print("mean drift of u", du, "of theta", dth, "worst point / bound", (err / bound).max())
    assert np.abs(du).max() < 1e-8 and abs(dth) < 3e-8
