"""The pointwise functions of the stage (csrc/dg_flux.cuh).  The reciprocal and the
square root of the FP64 stage: correctly rounded, bit for bit numpy's, over the whole
range of exponents and for zeros, subnormals, negative numbers, infinities and NaN.
The Rusanov flux: the bits of its definition with every rounding in its place,
whatever the compiler might contract at a call site."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2303_11767_gb300 import build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SOURCE = """
#include "dg_flux.cuh"
__global__ void apply(const double *x, double *r, double *s, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = dgk::rcp(x[i]), s[i] = dgk::wave_sqrt(x[i]);
}
template <typename T> __device__ void opaque(T *v, int n)   // values that the compiler cannot trace
{
    for (int i = 0; i < n; ++i) {
        volatile T t = v[i];
        v[i] = t;
    }
}
template <typename T> __device__ T add(T a, T b);
template <> __device__ double add(double a, double b) { return __dadd_rn(a, b); }
template <> __device__ float add(float a, float b) { return __fadd_rn(a, b); }

// per state pair: the two fluxes (lambda, theta) and the same from the parts
template <typename T>
__global__ void rusanov(const T *q, T *got, T *want, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const T href = T(5960), g = T(9.80616), c = T(0.37);
    const T *L = q + 6 * i, *R = L + 3;
    unsigned st = 0;
    dgk::rusanov_lam(L, R, href, g, c, got + 6 * i, st);
    dgk::rusanov_th(L, R, href, g, c, got + 6 * i + 3, st);
    for (int d = 0; d < 2; ++d) {
        T fl[4], fr[4];
        if (d == 0) dgk::lam_flux(L, href, g, fl, fl[3], st), dgk::lam_flux(R, href, g, fr, fr[3], st);
        else dgk::th_flux(L, href, g, fl, fl[3], st), dgk::th_flux(R, href, g, fr, fr[3], st);
        opaque(fl, 4);
        opaque(fr, 4);
        for (int f = 0; f < 3; ++f) {
            T sum = add(fl[f], fr[f]), jump = add(R[f], -L[f]);
            opaque(&sum, 1);
            want[6 * i + 3 * d + f] = T(0.5) * c * fma(-fmax(fl[3], fr[3]), jump, sum);
        }
    }
}
extern "C" int rusanov_f32(const float *q, float *got, float *want, int n)
{
    rusanov<<<(n + 255) / 256, 256>>>(q, got, want, n);
    return cudaDeviceSynchronize() != cudaSuccess;
}
extern "C" int rusanov_f64(const double *q, double *got, double *want, int n)
{
    rusanov<<<(n + 255) / 256, 256>>>(q, got, want, n);
    return cudaDeviceSynchronize() != cudaSuccess;
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


@pytest.fixture(scope="module")
def functions(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("flux")
    src, lib = tmp / "f.cu", tmp / "f.so"
    src.write_text(SOURCE)
    subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-I" + build.CSRC, "-shared", "-o", str(lib), str(src)], check=True,
                   env={**os.environ, "TMPDIR": str(tmp)})
    return ctypes.CDLL(str(lib))


def _call(fn, *tensors):
    torch.cuda.synchronize()
    assert fn(*[ctypes.c_void_p(t.data_ptr()) for t in tensors[:-1]], tensors[-1]) == 0


def test_correctly_rounded(functions):
    x = _arguments()
    dx = torch.from_numpy(x).cuda()
    r, s = torch.empty_like(dx), torch.empty_like(dx)
    _call(functions.flux_functions, dx, r, s, len(x))
    with np.errstate(all="ignore"):
        for got, want in ((r.cpu().numpy(), 1.0 / x), (s.cpu().numpy(), np.sqrt(x))):
            same = (got.view(np.int64) == want.view(np.int64)) | (np.isnan(got) & np.isnan(want))
            assert same.all(), (x[~same][:5], got[~same][:5], want[~same][:5], (~same).mean())


@pytest.mark.parametrize("name,dtype", [("rusanov_f32", np.float32), ("rusanov_f64", np.float64)])
def test_rusanov_rounds_as_defined(functions, name, dtype):
    rng = np.random.default_rng(2)
    n = 1 << 16
    q = (rng.normal(size=(n, 2, 3)) * [200.0, 1e5, 1e5]).astype(dtype)
    dq = torch.from_numpy(q).cuda()
    got, want = torch.zeros(n, 6, dtype=dq.dtype, device="cuda"), torch.ones(n, 6, dtype=dq.dtype, device="cuda")
    _call(getattr(functions, name), dq, got, want, n)
    assert torch.equal(got, want), (got != want).double().mean(0)
