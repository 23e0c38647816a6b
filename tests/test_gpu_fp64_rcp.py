"""The FP64 step's reciprocal (fp64::rcp) on the device: r rounded once from an estimate
whose own error is below 2^-60, so |1 - x r| is at most half a unit in the last place of 1
(2^-53) but for that error."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1802_02868_gb300 import build

pytestmark = pytest.mark.gpu


def test_reciprocal_over_the_range_of_exponents(tmp_path):
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("long double is double here")
    import torch
    src = tmp_path / "rcp.cu"
    src.write_text('#include "%s"\n'
                   "__global__ void k(const double *x, double *r, int n)\n"
                   "{\n"
                   "    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) r[i] = dugks::fp64::rcp(x[i]);\n"
                   "}\n"
                   'extern "C" int run(const double *x, double *r, int n)\n'
                   "{\n"
                   "    k<<<64, 256>>>(x, r, n);\n"
                   "    return (int)cudaDeviceSynchronize();\n"
                   "}\n" % os.path.join(build.CSRC, "dugks_fp64.cuh"))
    so = tmp_path / "rcp.so"
    subprocess.run([build.nvcc(), "-shared", str(src), "-o", str(so)] + build._flags() + ["-lcudart"], check=True,
                   stdout=subprocess.PIPE, stderr=subprocess.STDOUT)
    rng = np.random.default_rng(11)
    n = 1 << 20
    x = np.ldexp(1.0 + rng.random(n), rng.integers(-1000, 1001, n)) * rng.choice([-1.0, 1.0], n)
    x[:4] = 1.0, -1.0, np.nextafter(2.0, 1.0), np.nextafter(1.0, 2.0)
    dx = torch.from_numpy(x).cuda()
    dr = torch.empty_like(dx)
    torch.cuda.synchronize()
    run = ctypes.CDLL(str(so)).run
    run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    assert run(dx.data_ptr(), dr.data_ptr(), n) == 0
    e = np.abs(1 - x.astype(np.longdouble) * dr.cpu().numpy().astype(np.longdouble))
    assert float(e.max()) <= 2.0 ** -53 * (1 + 2.0 ** -6)
