"""The reciprocal on the integer pipe (1/T, 1/rho, pivots, error scales) is correctly rounded,
as the division it stands for: every value equals numpy's 1/x bit for bit."""
import ctypes as C

import numpy as np
import pytest

from paper_2508_16105_gb300 import build, rde_chem, synth


def arguments():
    """Mantissas over [1, 2) with small and large exponents, those whose reciprocals lie
    nearest to the middle between two doubles, and what the integer form leaves to division."""
    m = 1.0 + synth.uniform_range(51, "mantissa", 1 << 20, 0.0, 1.0)
    e = np.floor(synth.uniform_range(52, "exponent", m.size, -1022.0, 1024.0))
    # D = 2^106 / (2 q + 1) rounded: D's reciprocal is within half a unit of D from a midpoint
    q = (1 << 52) + (synth.uniform_range(53, "quotient", 1 << 16, 0.0, 1.0) * 2.0 ** 52).astype(np.int64)
    hard = np.array([float(((1 << 106) + int(v)) // (2 * int(v) + 1)) for v in q]) * 2.0 ** -53
    near = np.concatenate([2.0 - np.arange(1, 200) * 2.0 ** -52, 1.0 + np.arange(0, 200) * 2.0 ** -52])
    powers = np.ldexp(1.0, np.arange(-1074, 1024))
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, np.finfo(float).max])
    with np.errstate(over="ignore"):
        x = np.concatenate([np.ldexp(m, e.astype(int)), hard, near, powers, special])
    return np.concatenate([x, -x])


def function():
    build.build_library()
    lib = rde_chem.load_library()
    lib.rde_selftest_math.argtypes = [C.c_int, C.c_int64, C.c_void_p, C.c_void_p, C.c_int, C.c_void_p]
    return lib.rde_selftest_math


def check(x, y):
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / x
    bad = ~((y.view(np.int64) == want.view(np.int64)) | (np.isnan(y) & np.isnan(want)))
    assert not bad.any(), (int(bad.sum()), x[bad][:4], y[bad][:4], want[bad][:4])


def test_host():
    x = arguments()
    y = np.empty_like(x)
    assert function()(2, x.size, x.ctypes.data, y.ctypes.data, 0, None) == 0
    check(x, y)


@pytest.mark.gpu
def test_device():
    import torch
    x = arguments()
    dx = torch.as_tensor(x, device="cuda")
    dy = torch.empty_like(dx)
    assert function()(2, x.size, dx.data_ptr(), dy.data_ptr(), 1, torch.cuda.current_stream().cuda_stream) == 0
    check(x, dy.cpu().numpy())
