"""Spreading by strips (csrc/nufft_strip.cuh; FP64 plans with double-float weights) at every kernel support.

The deterministic plan of the same geometry spreads with FP64 taps, one point per thread, so the two adjoints must
agree to the 2e-12 that tests/test_gpu_parity.py allows them.  Points: uniform, all at one cell (long runs of
one row), poles and both ends of phi, few enough to leave most tiles empty; tile heights 16 to 64 and the default.
"""
import numpy as np
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


def points(kind):
    if kind == "few":
        th, ph, chi = W.random_points(19, 5)
    elif kind == "uniform":
        th, ph, chi = W.random_points(30011, 6)
    else:  # 2,000 points within one grid cell, and the domain's edges
        th, ph, chi = W.random_points(2017, 7)
        th, ph = 1.1 + 1e-4 * th, 6.2 + 1e-5 * ph
        th[:6] = [0.0, np.pi, 1e-9, np.pi - 1e-9, 0.5 * np.pi, 0.0]
        ph[:6] = [0.0, 2 * np.pi, 6.2831853, 0.0, np.pi, 3.0]
    return th, ph, chi


@pytest.mark.parametrize("w", range(4, 17))
@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("kind", ["few", "uniform", "cluster"])
def test_adjoint_equals_fp64_taps(w, spin, kind):
    th, ph, chi = points(kind)
    kw = dict(spin=spin, epsilon=1e-6, precision="fp64", sigma=2.0, W=w, device=DEV)
    y = torch.as_tensor(np.random.default_rng(w).standard_normal((1 if spin == 0 else 2, th.size)), device=DEV)
    y[:, ::7] *= 1e-3
    det = LensPlan(70, th, ph, chi, deterministic=True, **kw)
    ref = det.adjoint(y)
    for rows in (0, 16, 64):
        plan = LensPlan(70, th, ph, chi, spread_tile_rows=rows, **kw)
        got = plan.adjoint(y)
        assert float(torch.linalg.norm(got - ref) / torch.linalg.norm(ref)) <= 2e-12
        # the scale is exact (the Legendre step holds its inputs in FP32 pairs: within their range)
        for f in (2.0 ** 60, 2.0 ** -60):
            assert torch.equal(torch.isfinite(plan.adjoint(y * f)), torch.isfinite(got))
            assert float(torch.linalg.norm(plan.adjoint(y * f) / f - got) / torch.linalg.norm(got)) <= 1e-13
        z = y.clone()
        z[0, 3] = float("nan")
        assert bool(torch.isnan(plan.adjoint(z)).any())
        plan.close()
    assert float(torch.linalg.norm(LensPlan(70, th, ph, chi, **kw).adjoint(torch.zeros_like(y)))) == 0.0
    det.close()
