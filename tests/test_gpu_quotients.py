"""The FP64 quotients of bz_device.cuh (rcp64, div64, scaled_rcp) against correctly
rounded ones, and the reconstruction weights built on them where the smoothness
indicators leave the range of a plain reciprocal."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2103_14890_gb300 import build, workloads
from gpu_util import bz_module

pytestmark = pytest.mark.gpu

SOURCE = """
#include "bz_device.cuh"
__global__ void quotients(const double *a, const double *b, const int *scale, double *r, double *q, double *s, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = bz::rcp64(b[i]);
    q[i] = bz::div64(a[i], b[i], r[i]);
    s[i] = bz::scaled_rcp(b[i] < 0 ? -b[i] : b[i], scale[i]);
}
extern "C" int run(const double *a, const double *b, const int *scale, double *r, double *q, double *s, int n) {
    quotients<<<(n + 255) / 256, 256>>>(a, b, scale, r, q, s, n);
    return (int)cudaDeviceSynchronize();
}
"""


def _values(n):
    """Random mantissas and values next to powers of two, both signs, exponents -300 to 300."""
    rng = np.random.default_rng(8)
    m = rng.uniform(1.0, 2.0, n)
    near = 1.0 + 2.0 ** -52 * rng.integers(0, 64, n)
    m = np.where(np.arange(n) % 3 == 0, near, np.where(np.arange(n) % 3 == 1, m, 2.0 - (near - 1.0)))
    return m * np.exp2(rng.integers(-300, 301, n).astype(np.float64)) * rng.choice([-1.0, 1.0], n)


def test_quotients_against_correctly_rounded(tmp_path):
    import torch
    src = tmp_path / "q.cu"
    src.write_text(SOURCE)
    lib = tmp_path / "libq.so"
    subprocess.run([build._nvcc(), "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", *build.ARCH, "-I", build.CSRC,
                    str(src), "-o", str(lib)], check=True)
    n = 1 << 20
    a, b = _values(n)[::-1].copy(), _values(n)
    # 2^e at or below |b|, as the weights take it from the least indicator
    gap = np.random.default_rng(9).integers(0, 700, n)
    e = np.frexp(b)[1] - 1 - gap
    t = [torch.from_numpy(x).cuda() for x in (a, b, (e << 20).astype(np.int32))]
    out = [torch.empty(n, device="cuda", dtype=torch.float64) for _ in range(3)]
    torch.cuda.synchronize()
    rc = ctypes.CDLL(os.fspath(lib)).run(*[ctypes.c_void_p(x.data_ptr()) for x in t + out], n)
    assert rc == 0
    r, q, s = (x.cpu().numpy() for x in out)

    def ulps(x, y):                        # both finite and of one sign
        return np.abs(x.view(np.int64) - y.view(np.int64))

    # 2^-51 of the result is at most 4 ulp, its rounding and the reference's half an ulp each
    assert ulps(r, 1.0 / b).max() <= 5
    d = ulps(q, a / b)
    assert d.max() <= 1 and (d > 0).mean() < 1e-3, (d.max(), (d > 0).mean())
    want = np.exp2(e.astype(np.float64)) / np.abs(b)
    assert (want <= 1.0).all() and ulps(s, want).max() <= 5
    print("reciprocals: largest error %d ulp, quotients not correctly rounded: %.1e" % (ulps(r, 1.0 / b).max(), (d > 0).mean()))


@pytest.mark.parametrize("order", [2, 3])
def test_transport_of_large_values(order):
    """FP64 transport of data scaled by a power of two is the scaled residual, up to smoothness indicators just below
    overflow (at most 0.46 on this data, against which the weights' eps of 1e-14 is nothing from 2^100 on)."""
    import torch
    bz = bz_module()
    pts, cells = workloads.periodic_voronoi(60)
    m, g = bz.Mesh(pts, cells, order=order, periodic=(10.0, 10.0)), bz.Grid(2, 8, 6.0)
    f = torch.from_numpy(1.0 + 0.6 * np.random.default_rng(3).random((len(cells), 64))).cuda()

    def scaled(k):
        got = bz.transport_residual(m, g, torch.ldexp(f, torch.tensor(k)), precision="fp64")
        bz.check()
        return torch.ldexp(got, torch.tensor(-k))

    want = scaled(100)
    for k in (300, 505, 509, 511, 512):
        got = scaled(k)
        assert torch.isfinite(got).all() and float((got - want).abs().max() / want.abs().max()) < 1e-12, k
