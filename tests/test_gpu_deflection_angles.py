"""k_deflection_vjp (csrc/gradient.cu) on both of its branches: power series up to half a radian, closed forms above.

Deflections of 0.05 rad rms all take the series, 0.5 rad rms both, 1 rad rms mostly the closed forms; the oracle's
gradient is the reference, to the 1e-9 that tests/test_gpu_phi_gradient.py allows it.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2304_10431_gb300 import LensingModel
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


def potential(L, seed, rms):
    phi = W.draw_alm(W.phi_cl(L), L, seed)
    ell = W.alm_l_of_index(L).astype(float)
    w = np.where(W.alm_m_of_index(L) > 0, 2.0, 1.0)
    return phi * rms / np.sqrt(np.sum(w * ell * (ell + 1) * np.abs(phi) ** 2) / (4 * np.pi))


@pytest.mark.parametrize("spin", [0, 2])
@pytest.mark.parametrize("rms", [0.05, 0.5, 1.0])
def test_series_and_closed_forms(spin, rms):
    L = 32
    th0, ph0 = W.healpix_centres(8)
    phi = potential(L, 9, rms)
    x = np.stack([W.draw_alm(W.cmb_cl(L, 25.0), L, 30 + k, spin=spin) for k in range(1 if spin == 0 else 2)])
    g = np.random.default_rng(1).standard_normal((x.shape[0], th0.size))
    model = LensingModel(L, th0, ph0, spin=spin, epsilon=1e-12, precision="fp64", device=DEV)
    model.set_phi(torch.as_tensor(phi, device=DEV))
    a = model.alpha.norm(dim=0)
    assert bool((a <= 0.5).any()) and (rms < 0.2 or bool((a > 0.5).any()))
    got = model.grad_phi(torch.as_tensor(x, device=DEV), torch.as_tensor(g, device=DEV)).cpu().numpy()
    ref = O.phi_gradient(L, spin, th0, ph0, phi, L, x, g)
    assert np.linalg.norm(got - ref) <= 1e-9 * np.linalg.norm(ref)
    model.close()
