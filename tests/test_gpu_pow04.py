"""The contact area's power x^0.4 of the device code, compiled here into a kernel of its
own, against the power in extended precision, over the whole range that the function
takes itself and at its ends.  Bound: with u = 2^-53, x^2 / y^5 carries at most six
roundings (6 u, a fifth of it in the result) and the last sum one: 2.2 u < 2.5e-16."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = """
#include "particle_math.cuh"
__global__ void k_pow04(const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = tribo::pow04(x[i]);
}
extern "C" int run_pow04(const double* x, double* y, int n) {
    k_pow04<<<(n + 255) / 256, 256>>>(x, y, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_power_is_rounded_from_extended_precision(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_10761_gb300 import build
    src, lib = str(tmp_path / "pow04.cu"), str(tmp_path / "libpow04.so")
    with open(src, "w") as fh:
        fh.write(SOURCE)
    r = subprocess.run([build.nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-I" + build.CSRC, "-shared", src, "-o", lib, "-lcudart"],
                       capture_output=True, text=True)
    assert r.returncode == 0 and os.path.exists(lib), r.stderr
    rng = np.random.default_rng(4)
    x = np.concatenate([10.0 ** rng.uniform(-30, 30, 1 << 20), 10.0 ** rng.uniform(-9, -3, 1 << 20),
                        np.nextafter(1e-30, 1) * np.ones(1), np.nextafter(1e30, 1) * np.ones(1), [1e-30, 1e30, 1.0, 1e-300, 1e300]])
    xd = torch.from_numpy(x).cuda()
    yd = torch.empty_like(xd)
    torch.cuda.synchronize()
    run = ctypes.CDLL(lib).run_pow04
    run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    assert run(xd.data_ptr(), yd.data_ptr(), x.size) == 0
    ref = np.power(x.astype(np.longdouble), np.longdouble(0.4))
    err = np.abs((yd.cpu().numpy().astype(np.longdouble) - ref) / ref).astype(np.float64)
    own = (x > 1e-30) & (x < 1e30)
    assert err[own].max() <= 2.5e-16
    assert err[~own].max() <= 4.5e-16          # CUDA's pow: two units in the last place
