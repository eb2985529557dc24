"""FP64 adjoints over the exponent range of doubles.

Spreading by strips scales each tile by a power of two, so a map times 2^k has the a_lm times 2^k.  Plans below lmax 256
run the Legendre step in native FP64 and keep that range to their a_lm; only the order of the atomic sums differs between
two calls (1e-13, as tests/test_gpu_strip.py allows them).
"""
import numpy as np
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("k", [-900, -600, 600, 900])
def test_adjoint_scales_with_the_map(spin, k):
    th, ph, chi = W.random_points(5003, 8)
    plan = LensPlan(70, th, ph, chi, spin=spin, epsilon=1e-10, precision="fp64", device=DEV)
    y = torch.as_tensor(np.random.default_rng(3).standard_normal((1 if spin == 0 else 2, th.size)), device=DEV)
    ref = plan.adjoint(y)
    got = plan.adjoint(y * 2.0 ** k) * 2.0 ** -k
    assert float(torch.linalg.norm(got - ref) / torch.linalg.norm(ref)) <= 1e-13
