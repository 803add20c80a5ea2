"""The sum of squares that the FP64 residual pass takes of its FP32 copy."""
import ctypes
import os
import subprocess

import pytest

from paper_1611_09638_gb300 import build as B

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("shape", [(64, 64, 64), (256, 256, 512), (512, 512, 512)])
def test_sum_of_squares_of_any_length(tmp_path, shape):
    """A constant residual whose square drifts by 1.2e-5 where 862 of them are
    summed in FP32 (a thread's share of 512^3): FP32 sums of 64 terms are
    within 64 x 2^-24."""
    lib = str(tmp_path / "residual_norm.so")
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-shared", "-o", lib, os.path.join(HERE, "host", "residual_norm.cu")],
                   check=True)
    L = ctypes.CDLL(lib)
    value = 1.4128963947296143
    u, ones = torch.zeros(shape, device="cuda", dtype=torch.float64), torch.ones(shape, device="cuda", dtype=torch.float64)
    f, F = ones * value, torch.ones((3, *shape), device="cuda", dtype=torch.float64)
    r32 = torch.empty(shape, device="cuda", dtype=torch.float32)
    part = torch.empty(L.partials(), device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    rc = L.residual_partials(*shape, *(ctypes.c_void_p(t.data_ptr()) for t in (u, f, F, ones, r32, part)))
    assert rc == 0
    assert torch.all(r32 == value)
    assert abs(part.sum().item() / (u.numel() * value ** 2) - 1.0) <= 64 * 2.0 ** -24
