"""The reciprocal and the square root of the FP64 stage (csrc/dg_flux.cuh): correctly
rounded, bit for bit numpy's, over the whole range of exponents and for zeros,
subnormals, negative numbers, infinities and NaN."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_11767_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "dg_flux.cuh"
__global__ void apply(const double *x, double *r, double *s, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = dgk::rcp(x[i]), s[i] = dgk::wave_sqrt(x[i]);
}
extern "C" int flux_functions(const double *x, double *r, double *s, int n)
{
    apply<<<(n + 255) / 256, 256>>>(x, r, s, n);
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


def _arguments():
    rng = np.random.default_rng(1)
    m = 1.0 + rng.integers(0, 2 ** 52, 2 ** 20) * 2.0 ** -52
    x = np.concatenate([np.ldexp(m, rng.integers(-1022, 1024, m.size)), m, 6000.0 * m])
    e = np.arange(-1074, 1024)
    powers = np.ldexp(1.0, e)
    ends = np.array([0.0, 5e-324, 2.2e-308, np.finfo(float).max, np.inf, np.nan])
    near = np.concatenate([np.nextafter(powers, 0), powers, np.nextafter(powers, np.inf)])
    return np.concatenate([x, near, ends, -x[:1000], -near, -ends])


def test_correctly_rounded(tmp_path):
    torch = pytest.importorskip("torch")
    src, lib = tmp_path / "f.cu", tmp_path / "f.so"
    src.write_text(SOURCE)
    subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-I" + build.CSRC, "-shared", "-o", str(lib), str(src)], check=True,
                   env={**os.environ, "TMPDIR": str(tmp_path)})
    x = _arguments()
    dx = torch.from_numpy(x).cuda()
    r, s = torch.empty_like(dx), torch.empty_like(dx)
    p = [ctypes.c_void_p(t.data_ptr()) for t in (dx, r, s)]
    torch.cuda.synchronize()
    assert ctypes.CDLL(str(lib)).flux_functions(*p, len(x)) == 0
    with np.errstate(all="ignore"):
        for got, want in ((r.cpu().numpy(), 1.0 / x), (s.cpu().numpy(), np.sqrt(x))):
            same = (got.view(np.int64) == want.view(np.int64)) | (np.isnan(got) & np.isnan(want))
            assert same.all(), (x[~same][:5], got[~same][:5], want[~same][:5], (~same).mean())
