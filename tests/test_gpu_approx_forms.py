"""The single-instruction division and square root of the collisions and wall laws
against the full-range forms (div_cell, sqrt_cell), bit for bit over the operands for
which they stand in for each other: every mantissa of a divisor or radicand, and
random pairs whose operands and quotient are normal numbers."""
import ctypes
import subprocess

import numpy as np
import pytest
import torch

from paper_2009_04352_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_device.cuh"

__global__ void k_forms(const float *a, const float *b, int n, float *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = lbm::div_cell<false>(a[i], b[i]);
    out[n + i] = lbm::div_cell<true>(a[i], b[i]);
    out[2 * n + i] = lbm::sqrt_cell<false>(fabsf(b[i]));
    out[3 * n + i] = lbm::sqrt_cell<true>(fabsf(b[i]));
}

extern "C" int run_forms(const float *a, const float *b, int n, float *out)
{
    k_forms<<<(n + 255) / 256, 256>>>(a, b, n, out);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def forms(tmp_path_factory):
    d = tmp_path_factory.mktemp("forms")
    (d / "forms.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.FLAGS, "-I" + build.CSRC, "-shared", "-o", str(d / "forms.so"), str(d / "forms.cu")],
                   check=True)
    fn = ctypes.CDLL(str(d / "forms.so")).run_forms
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def run(a, b):
        a, b = (torch.from_numpy(v).cuda() for v in (a, b))
        out = torch.empty(4 * a.numel(), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        assert fn(a.data_ptr(), b.data_ptr(), a.numel(), out.data_ptr()) == 0
        return out.view(torch.int32).view(4, -1)
    return run


def _same(forms, a, b):
    got = forms(a, b)
    assert torch.equal(got[0], got[1])
    assert torch.equal(got[2], got[3])


@pytest.mark.parametrize("numerator", [2.0, -1.0, 1e-3, -3e-7, 0.7853982, 0.0])
@pytest.mark.parametrize("exponent", [-40, -2, -1, 0, 1, 2, 60])
def test_every_mantissa_of_the_divisor(forms, exponent, numerator):
    b = np.ldexp((1 << 23) + np.arange(1 << 23, dtype=np.float64), exponent - 23).astype(np.float32)
    _same(forms, np.full_like(b, numerator), b)


def test_normal_operands_and_quotients(forms):
    r = np.random.RandomState(2)
    n = 1 << 24
    b = np.ldexp(1.0 + r.rand(n), r.randint(-100, 101, n)).astype(np.float32) * r.choice([-1.0, 1.0], n).astype(np.float32)
    q = np.ldexp(1.0 + r.rand(n), r.randint(-125, 126, n))
    with np.errstate(over="ignore", under="ignore"):
        a = (q * b).astype(np.float32)
    keep = (np.abs(a) >= 2.0 ** -125) & (np.abs(a) < 2.0 ** 125)
    assert keep.sum() > n // 4
    _same(forms, a[keep], b[keep])


def test_relaxation_and_velocity_operands(forms):
    """-(rho - 1) / rho and 2 / (tau0 + sqrt(tau0^2 + c q)) at densities and rates of channels."""
    r = np.random.RandomState(3)
    n = 1 << 24
    d = (r.choice([-1.0, 1.0], n) * 10.0 ** r.uniform(-9, -0.3, n)).astype(np.float32)
    _same(forms, -d, np.float32(1) + d)
    tau = (0.5 + 10.0 ** r.uniform(-6, 1, n)).astype(np.float32)
    _same(forms, np.full(n, 2.0, np.float32), tau + np.sqrt(tau * tau + (10.0 ** r.uniform(-30, 0, n)).astype(np.float32)))
