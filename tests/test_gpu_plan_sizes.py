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
