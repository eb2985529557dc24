"""FP64 interpolation with double-float weights (csrc/nufft.cuh, k_interp_dd) at every kernel support.

The plan without the point-weight table interpolates with FP64 taps; tests/test_gpu_parity.py allows the two 1e-12.
Point counts around a warp's 32 and a block's 128, whose last warp stages fewer weights.
"""
import numpy as np
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("w", range(4, 17))
@pytest.mark.parametrize("spin", [0, 2])
def test_synthesis_equals_fp64_taps(w, spin):
    L = 70
    rng = np.random.default_rng(w)
    for n in (1, 31, 33, 127, 129, 5003):
        th, ph, chi = W.random_points(n, 3 + n)
        th[0], ph[0] = 0.0, 2 * np.pi
        kw = dict(spin=spin, epsilon=1e-6, precision="fp64", sigma=2.0, W=w, device=DEV)
        table = LensPlan(L, th, ph, chi, point_weights=1, **kw)
        taps = LensPlan(L, th, ph, chi, point_weights=-1, **kw)
        nc, nalm = (1 if spin == 0 else 2), (L + 1) * (L + 2) // 2
        a = rng.standard_normal((nc, nalm)) + 1j * rng.standard_normal((nc, nalm))
        a = torch.as_tensor(a, device=DEV)
        got, ref = table.synthesis(a), taps.synthesis(a)
        assert float(torch.linalg.norm(got - ref) / torch.linalg.norm(ref)) <= 1e-12
