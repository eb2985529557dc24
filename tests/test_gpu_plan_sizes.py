"""Sizes a plan reports are those it allocates."""
import pytest
import torch

from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


@pytest.mark.parametrize("w", [12, 13])
@pytest.mark.parametrize("eps", [1e-9, 1e-11])  # weights as double-float pairs, as doubles
def test_point_weight_bytes(w, eps):
    info = []
    for n in (4001, 9001):
        th, ph, _ = W.random_points(n, 3)
        info.append(LensPlan(300, th, ph, epsilon=eps, precision="fp64", sigma=2.0, W=w, device=DEV).info())
    # per point: first cell and index (4 bytes each), offsets (two doubles), weights
    grown = [b - a for a, b in ((info[0][k], info[1][k]) for k in ("plan_bytes", "point_weight_bytes"))]
    assert grown[0] == 24 * 5000 + grown[1] and grown[1] == 16 * w * 5000


@pytest.mark.parametrize("restart", [0, -1])
def test_grouped_synthesis_workspace(restart):
    """Four maps in one call: four sets of ring coefficients, and of prepared a_lm only where the kernels read them
    (plans without restart values)."""
    th, ph, chi = W.random_points(4001, 3)
    plan = LensPlan(64, th, ph, chi, spin=2, epsilon=1e-5, legendre_restart=restart, device=DEV)
    before = plan.info()
    plan.synthesis(torch.zeros(4, 2, plan.nalm, dtype=plan.complex_dtype, device=DEV))
    rings = 4 * 8 * (2 * 64 + 1) * before["ntheta"]
    grown = plan.info()["workspace_bytes"] - before["workspace_bytes"]
    assert grown == rings + (0 if restart == 0 else 4 * 8 * 2 * plan.nalm)
