"""FP64 plans with restart values (double-float Legendre steps and, where deconvolution allows it, double-float synthesis
transforms) against the all-FP64 plan of the same sigma and W: the error of a synthesis, measured against a plan of epsilon
1e-13, must not grow.

Both plans make the same truncation error, far above their rounding: the restarted recursion's (about 3e-12 of the
map) changes the error of 1e-10 and more by less than 5e-4 of itself, hence the bound 1.001.  W 16 at sigma 1.2 amplifies
rounding most among the choices of plan creation (8e6 over both axes), W 13 at 1.6 is the usual choice.
"""
import numpy as np
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("sigma,w,eps", [(1.2, 16, 1e-8), (1.3, 15, 1e-9), (1.6, 11, 1e-8)])
def test_error_is_that_of_fp64_transforms(spin, sigma, w, eps):
    L = 400
    th, ph, chi = W.random_points(50021, 4)
    kw = dict(spin=spin, precision="fp64", device=DEV)
    native = dict(legendre_restart=-1, legendre_df32_mmin=-1)
    rng = np.random.default_rng(w)
    nalm = (L + 1) * (L + 2) // 2
    a = rng.standard_normal((1 if spin == 0 else 2, nalm)) + 1j * rng.standard_normal((1 if spin == 0 else 2, nalm))
    a = torch.as_tensor(a, device=DEV)
    ref = LensPlan(L, th, ph, chi, epsilon=1e-13, **native, **kw).synthesis(a)
    err = [float(torch.linalg.norm(LensPlan(L, th, ph, chi, epsilon=eps, sigma=sigma, W=w, **x, **kw).synthesis(a) - ref))
           for x in ({}, native)]
    assert err[0] <= 1.001 * err[1]
