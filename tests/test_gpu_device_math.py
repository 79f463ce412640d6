"""The reciprocal square root and square root that the Lanczos scalars use
(csrc/kg_internal.h), compiled on their own, over FP64's exponents and the
mantissas where their steps change.

Tolerance of rsqrt3, 2^-52 relative: half a unit of the last rounding and a
quarter from the rounded product in r, the series' remainder (5/16) r^3 being
below 2^-61 for a starting value with |r| < 2^-20.  Of sqrt_from, 2^-52: Newton's
correction leaves the last rounding.  CUDA's own rsqrt and sqrt have to agree to
the sum of both errors, 2^-51.
"""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_1109_1205_gb300 import build  # noqa: E402

SOURCE = r"""
#include "kg_internal.h"
__global__ void roots(const double* x, int n, double* out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double r = kg::rsqrt3(x[i]);
    out[i] = r;
    out[n + i] = kg::sqrt_from(x[i], r);
    out[2 * n + i] = rsqrt(x[i]);
    out[3 * n + i] = sqrt(x[i]);
}
extern "C" int run_roots(const double* x, int n, double* out) {
    roots<<<(n + 127) / 128, 128>>>(x, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


def test_roots(tmp_path):
    src, lib = tmp_path / "roots.cu", tmp_path / "roots.so"
    src.write_text(SOURCE)
    subprocess.check_call([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", str(src), "-o", str(lib)])
    rng = np.random.default_rng(3)
    mant = np.concatenate([1.0 + rng.random(20000) * 3.0, 1.0 + 2.0 ** -np.arange(1, 53), 2.0 - 2.0 ** -np.arange(0, 53),
                           4.0 - 2.0 ** -np.arange(0, 52), [1.0, 2.0, 3.0]])
    x = np.concatenate([mant * 2.0 ** rng.integers(-500, 500, mant.size) * 2.0 ** rng.integers(-500, 500, mant.size),
                        mant, [2.0 ** -1022, 2.0 ** 1023, 2.0 ** 1023 * (2 - 2.0 ** -52)]])
    xd = torch.from_numpy(x).cuda()
    out = torch.empty(4 * x.size, dtype=torch.float64, device="cuda")
    f = ctypes.CDLL(str(lib)).run_roots
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    torch.cuda.synchronize()
    assert f(xd.data_ptr(), x.size, out.data_ptr()) == 0
    r, b, cr, cb = out.cpu().numpy().reshape(4, -1).astype(np.longdouble)
    root = np.sqrt(x.astype(np.longdouble))
    assert np.max(np.abs(r * root - 1)) <= 2.0 ** -52
    assert np.max(np.abs(b / root - 1)) <= 2.0 ** -52
    assert np.max(np.abs(r / cr - 1)) <= 2.0 ** -51 and np.max(np.abs(b / cb - 1)) <= 2.0 ** -51
