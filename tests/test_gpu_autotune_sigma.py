"""FP32 plans of the autotuner: two adjoints of a white map agree to the 1e-6 that tests/test_gpu_batch.py allows."""
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan, autotune
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("lmax,n", [(256, 20000), (512, 200000)])
def test_fp32_adjoints_agree(lmax, n, spin):
    th, ph, chi = W.random_points(n, lmax)
    best = autotune(lmax, th, ph, chi, spin=spin, epsilon=1e-5, precision="fp32", reps=1, device=DEV, cache=False)
    assert best["sigma"] >= 1.4
    kw = {k: v for k, v in best.items() if k not in ("ms", "cached")}
    plan = LensPlan(lmax, th, ph, chi, spin=spin, epsilon=1e-5, precision="fp32", device=DEV, **kw)
    y = torch.randn(plan.ncomp, n, device=DEV)
    a = plan.adjoint(y)
    assert float(torch.linalg.norm(plan.adjoint(y) - a) / torch.linalg.norm(a)) <= 1e-6
