"""FP32 spreading by strips (csrc/nufft_strip.cuh, k_spread_strip32) at every kernel support, and tiles that several warps
share in both precisions.

The deterministic plan of the same geometry, kernel and later stages adds the same FP32 taps as 64-bit integers, so the two
adjoints differ by the strips' running FP32 sums alone: about sqrt(n / 3) 2^-25 of a sum of n terms of one sign, 1.6e-6 for
8192 points of a warp, more than any sweeps here, below the plans' epsilon of 5e-6.  FP64: the 2e-12 of
tests/test_gpu_strip.py.  Below epsilon 1e-5 every W spreads by strips; at 1e-5 W >= 10 does for every spin.
"""
import numpy as np
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


def error(th, ph, chi, y, rows, **kw):
    det, plan = LensPlan(70, th, ph, chi, deterministic=True, **kw), LensPlan(70, th, ph, chi, spread_tile_rows=rows, **kw)
    y = torch.as_tensor(y, dtype=plan.real_dtype, device=DEV)
    ref, got = det.adjoint(y), plan.adjoint(y)
    assert float(torch.linalg.norm(plan.adjoint(torch.zeros_like(y)))) == 0.0
    z = y.clone()
    z[0, -1] = float("nan")
    assert bool(torch.isnan(torch.view_as_real(plan.adjoint(z))).any())
    return float(torch.linalg.norm(got - ref) / torch.linalg.norm(ref))


@pytest.mark.parametrize("w", range(4, 17))
@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 65, 30011])
def test_adjoint_equals_deterministic(w, spin, n):
    th, ph, chi = W.random_points(n, 5)
    th[0], ph[0] = 0.0, 2 * np.pi
    th[-1] = np.pi
    y = np.random.default_rng(w).standard_normal((1 if spin == 0 else 2, n))
    for rows in (0, 16, 64):
        for eps in (5e-6,) if w < 10 else (5e-6, 1e-5):
            assert error(th, ph, chi, y, rows, spin=spin, epsilon=eps, sigma=2.0, W=w, device=DEV) <= 5e-6


@pytest.mark.parametrize("precision,w,eps,tol", [("fp32", 5, 5e-6, 5e-6), ("fp32", 8, 5e-6, 5e-6), ("fp32", 13, 1e-5, 5e-6),
                                                 ("fp64", 8, 1e-6, 2e-12), ("fp64", 13, 1e-6, 2e-12)])
@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("n", [4095, 4097, 5003, 300007])  # few parts, and more points than the parts of 128 hold
@pytest.mark.parametrize("spread", [1e-4, 0.05])  # one cell; rows and columns of a tile
def test_tiles_shared_by_warps(precision, w, eps, tol, spin, n, spread):
    th, ph, _ = W.random_points(n, 7)
    th, ph = 1.1 + spread * th / np.pi, 6.2 + 0.1 * spread * ph
    y = np.abs(np.random.default_rng(n).standard_normal((1 if spin == 0 else 2, n)))
    assert error(th, ph, None, y, 0, spin=spin, epsilon=eps, precision=precision, sigma=2.0, W=w, device=DEV) <= tol
