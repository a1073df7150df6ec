"""recip and rsqrt_iter (csrc/approx64.cuh) on their own, compiled into a small kernel:
every exponent with random mantissas, powers of two and their neighbours, the exponents
where recip divides instead, both signs, and the special values.

Bounds, in units in the last place of the result: recip's last step is one fused
update of a value good to 2^-40 or better, so its own rounding and no more than 2^-20
beside it: 0.51. rsqrt_iter: the rounding of x y (2^-53 of e, half of that in the
result), the next term of the series (2^-57) and its own rounding: 1.1."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
#include <stdint.h>
#include "approx64.cuh"
__global__ void run(const double *x, double *r, double *s, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = fil::recip(x[i]);
    s[i] = x[i] >= 1e-290 && x[i] <= 1.7976931348623157e308 ? fil::rsqrt_iter(x[i]) : 0.0;
}
extern "C" int approx64(const double *x, double *r, double *s, int n) {
    run<<<(n + 255) / 256, 256>>>(x, r, s, n);
    if (cudaGetLastError() != cudaSuccess) return 1;
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


def _on_device(tmp_path, x):
    from paper_1903_12609_gb300 import build
    src, lib = tmp_path / "a.cu", tmp_path / "a.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-I" + build.CSRC, str(src), "-o", str(lib)], check=True)
    xd = torch.from_numpy(x).cuda()
    r, s = torch.empty_like(xd), torch.empty_like(xd)
    torch.cuda.synchronize()
    f = ctypes.CDLL(str(lib)).approx64
    f.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    assert f(xd.data_ptr(), r.data_ptr(), s.data_ptr(), len(x)) == 0
    return r.cpu().numpy(), s.cpu().numpy()


def test_reciprocals_and_square_roots(tmp_path):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no long double wider than FP64")
    rng = np.random.default_rng(0)
    e = np.arange(-1074, 1024)
    m = np.concatenate([np.ones((len(e), 1)), rng.uniform(1, 2, (len(e), 60)),
                        np.full((len(e), 1), 1 + 2.0 ** -52), np.full((len(e), 1), 2 - 2.0 ** -52)], 1)
    x = np.ldexp(m, e[:, None]).ravel()
    x = np.concatenate([x, -x, [0.0, -0.0, np.inf, -np.inf, np.nan, 1e-290]])
    r, s = _on_device(tmp_path, x)
    with np.errstate(all="ignore"):
        special = ~np.isfinite(x) | (x == 0) | ~np.isfinite(1.0 / x)
        np.testing.assert_array_equal(r[special], (1.0 / x)[special])
        xl = x[~special].astype(np.longdouble)
        err = np.abs(r[~special].astype(np.longdouble) - 1 / xl)
        ulp = np.spacing(np.abs((1.0 / x)[~special])).astype(np.longdouble)
        assert np.all(err <= 0.51 * ulp)
        ok = (x >= 1e-290) & np.isfinite(x)
        exact = 1 / np.sqrt(x[ok].astype(np.longdouble))
        assert np.all(np.abs(s[ok].astype(np.longdouble) - exact) <=
                      1.1 * np.spacing(exact.astype(np.float64)).astype(np.longdouble))
