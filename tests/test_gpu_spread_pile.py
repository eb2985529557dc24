"""Integer spreading tiles (FP32 plans with W 7, FP64 plans below epsilon 5e-11) with far more points in one grid cell than
the tile's bound of 65535 counts, against the deterministic plan, whose grid sums are 64-bit.

A map of ones makes every partial sum as large as it can be; random signs leave sums far below the bound of their terms.
FP32: the plan's epsilon; FP64: the 2e-12 that tests/test_gpu_parity.py allows the two adjoints.
"""
import numpy as np
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("precision,eps,w,tol", [("fp32", 1e-5, 7, 1e-5), ("fp64", 1e-11, 15, 2e-12)])
@pytest.mark.parametrize("n", [2047, 2049, 65537, 150001])
def test_many_points_in_one_cell(spin, precision, eps, w, tol, n):
    th, ph, _ = W.random_points(n, 7)
    th, ph = 1.1 + 1e-4 * th, 6.2 + 1e-5 * ph
    th[:3], ph[:3] = [0.0, np.pi, 0.5 * np.pi], [0.0, 2 * np.pi, np.pi]
    kw = dict(spin=spin, epsilon=eps, precision=precision, sigma=2.0, W=w, device=DEV)
    plan, det = LensPlan(70, th, ph, **kw), LensPlan(70, th, ph, deterministic=True, **kw)
    y = torch.as_tensor(np.random.default_rng(n).standard_normal((1 if spin == 0 else 2, n)), dtype=plan.real_dtype, device=DEV)
    for m in (torch.ones_like(y), y):
        ref = det.adjoint(m)
        assert float(torch.linalg.norm(plan.adjoint(m) - ref) / torch.linalg.norm(ref)) <= tol
