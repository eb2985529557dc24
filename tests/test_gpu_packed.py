"""Packed Legendre kernels (csrc/legendre_pk.cuh) at the edges of their blocks and stages.

The kernels run 8-degree blocks, stage 64 degrees at a time, give a warp 32 x (rings per thread)
rings and pad the last block with zeros: band limits around those sizes, mmax < lmax, every spin
variant and rings-per-thread setting, against the oracle's Legendre functions.  FP32 plans:
2e-6, the tolerance of the restarted recursion's tests.  FP64 plans (double-float, a short restart
interval so that restarts happen): 5e-12, likewise.
"""
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2304_10431_gb300 import LensPlan
from paper_2304_10431_gb300 import workloads as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0") if torch.cuda.is_available() else None


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


def ring_adjoint_ref(L, M, spin, nt, r, grad):
    """The transpose of the ring synthesis from the oracle's Legendre functions."""
    nalm = W.nalm(L, M)
    out = np.zeros((1 if spin == 0 or grad else 2, nalm), complex)
    lam = {sg: np.stack([np.stack([O.slambda(L, m, sg, math.pi * j / (nt - 1)) for j in range(nt)])
                         for m in range(M + 1)]) for sg in {spin, -spin}}  # [m][ring][l]
    for m in range(M + 1):
        i = m * (2 * L + 1 - m) // 2 + np.arange(m, L + 1)
        if spin == 0:
            out[0, i] = r[m] @ lam[0][m][:, m:]
            continue
        u, v = r[M + m] @ lam[spin][m][:, m:], r[M - m] @ lam[-spin][m][:, m:]
        v = (-1) ** spin * v.conj()
        out[0, i] = -0.5 * (u + v)
        if not grad:
            out[1, i] = 0.5j * (u - v)
    return out


CASES = [(1, 1, 0), (8, 8, 0), (9, 9, 1), (10, 5, 2), (63, 63, 0), (64, 64, 2), (65, 40, 0), (72, 72, 3), (73, 73, 2),
         (130, 130, 0), (137, 137, 1)]


@pytest.mark.parametrize("L,M,spin", CASES)
@pytest.mark.parametrize("rpt", [1, 2, 4])
@pytest.mark.parametrize("grad", [False, True])
def test_fp32_block_edges(L, M, spin, rpt, grad):
    if grad and spin == 0:
        pytest.skip("gradient-only plans have spin > 0")
    check(L, M, spin, grad, "fp32", 2e-6, epsilon=1e-5, legendre_rpt=(rpt, rpt), legendre_restart=8 if L < 70 else 0)


@pytest.mark.parametrize("L,M,spin", [(300, 300, 0), (300, 280, 2), (321, 321, 1)])
@pytest.mark.parametrize("rpt", [1, 2])
@pytest.mark.parametrize("grad", [False, True])
def test_fp64_block_edges(L, M, spin, rpt, grad):
    if grad and spin == 0:
        pytest.skip("gradient-only plans have spin > 0")
    check(L, M, spin, grad, "fp64", 5e-12, epsilon=1e-10, legendre_rpt=(rpt, rpt))


def check(L, M, spin, grad, prec, tol, **kw):
    th, ph, chi = W.random_points(10, 3)
    plan = LensPlan(L, th, ph, chi, spin=spin, mmax=M, precision=prec, grad_only=grad, device=DEV, **kw)
    inf = plan.info()
    assert inf["legendre_restart"] > 0
    nt, nc = inf["ntheta"], plan.alm_ncomp
    cl = W.cmb_cl(L, 0.8 * L)
    a = np.stack([W.draw_alm(cl, L, 5 + k, mmax=M, spin=spin) for k in range(nc)])
    full = a if nc == (1 if spin == 0 else 2) else np.concatenate([a, np.zeros_like(a)])
    ring = plan.ring_synthesis(torch.as_tensor(a, dtype=plan.complex_dtype, device=DEV)).cpu().numpy()
    ref = O.ring_coeffs(L, M, spin, math.pi * np.arange(nt) / (nt - 1), full).T
    assert ring.shape == ref.shape and rel(ring, ref) < tol
    rng = np.random.default_rng(4)
    r = rng.standard_normal(ref.shape) + 1j * rng.standard_normal(ref.shape)
    if spin == 0:
        r[0] = r[0].real
    else:
        r[M] = r[M].real + 0j  # order 0: U and V of one column
    r = r.astype(np.complex64 if prec == "fp32" else np.complex128)
    got = plan.ring_adjoint(torch.as_tensor(r, dtype=plan.complex_dtype, device=DEV)).cpu().numpy()
    want = ring_adjoint_ref(L, M, spin, nt, r.astype(complex), grad)
    m0 = np.arange(L + 1)  # order 0 comes back real
    want[:, m0] = want[:, m0].real
    assert rel(got, want) < tol
    plan.close()
