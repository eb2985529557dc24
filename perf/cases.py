"""Measured workloads of the lensing transforms, through the Python binding.

Each case is one call (or one training step) that a CMB-lensing program makes on a plan it keeps:
forward lensing (a_lm -> values at deflected points), its adjoint, many maps of one geometry in one
call, and a gradient step with respect to the unlensed field and the lensing potential.  Inputs are
the shapes of the paper's workloads: Gaussian a_lm with a damped CMB-like spectrum, HEALPix ring
centres displaced by 2.5 arcmin (or points drawn uniformly on the sphere), white-noise maps for the
adjoint.  Everything is generated on the device from the seed.

A case holds
  op       "forward" | "adjoint" | "grad"
  spin     0 (temperature), 1 (deflection), 2 (polarisation), 3
  lmax, mmax, precision ("fp32" | "fp64"), epsilon
  nside    points: 12 nside^2 displaced HEALPix centres (0: npoints uniform on the sphere)
  npoints  with nside = 0
  nmaps    maps of the one geometry in the call (forward / adjoint)
"""
import math

import numpy as np
import torch

from paper_2304_10431_gb300 import LensingModel, LensPlan, lensed

ARCMIN = math.pi / 10800.0


def _case(name, op, spin, lmax, precision, epsilon, nside=0, npoints=0, mmax=None, nmaps=1):
    return {"name": name, "op": op, "spin": spin, "lmax": lmax, "mmax": lmax if mmax is None else mmax,
            "precision": precision, "epsilon": epsilon, "nside": nside, "npoints": npoints, "nmaps": nmaps}


def listed():
    return [
        # small maps in a loop over patches, realisations or tests: latency and launches count
        _case("t_fp32_l128_fwd", "forward", 0, 128, "fp32", 1e-5, nside=64),
        # the small FP64 temperature configuration (lmax 128, Nside 64, 1e-10), backwards
        _case("t_fp64_l128_adj", "adjoint", 0, 128, "fp64", 1e-10, nside=64),
        # polarisation at low resolution: large-scale B modes, quick simulations
        _case("eb_fp32_l512_fwd", "forward", 2, 512, "fp32", 1e-5, nside=256),
        # a catalogue of positions rather than a pixelisation: odd counts, mmax < lmax, looser accuracy
        _case("t_fp32_l777_adj_ragged", "adjoint", 0, 777, "fp32", 1e-4, npoints=1000003, mmax=701),
        # a batch of simulated temperature maps lensed by one potential
        _case("t_fp32_l1024_32maps_fwd", "forward", 0, 1024, "fp32", 1e-5, nside=512, nmaps=32),
        # one step of a gradient-based fit of E/B and the potential: lensed map, both gradients
        _case("eb_fp32_l1024_grad", "grad", 2, 1024, "fp32", 1e-5, nside=512),
        # the polarisation configuration (lmax 2048, Nside 1024): adjoint in FP32, forward in FP64
        _case("eb_fp32_l2048_adj", "adjoint", 2, 2048, "fp32", 1e-5, nside=1024),
        _case("eb_fp64_l2048_fwd", "forward", 2, 2048, "fp64", 1e-10, nside=1024),
        # the headline size (lmax 4096, Nside 2048, 50.3M points): T and E/B forward, E/B adjoint
        _case("t_fp32_l4096_fwd", "forward", 0, 4096, "fp32", 1e-5, nside=2048),
        _case("eb_fp32_l4096_fwd", "forward", 2, 4096, "fp32", 1e-5, nside=2048),
        _case("eb_fp32_l4096_adj", "adjoint", 2, 4096, "fp32", 1e-5, nside=2048),
        # the same size in FP64, temperature, backwards
        _case("t_fp64_l4096_adj", "adjoint", 0, 4096, "fp64", 1e-10, nside=2048),
    ]


def draw(rng):
    precision = rng.choice(["fp32", "fp32", "fp64"])
    epsilon = rng.choice([1e-4, 1e-5, 1e-5] if precision == "fp32" else [1e-6, 1e-8, 1e-9, 1e-10, 1e-10])
    op = rng.choice(["forward"] * 4 + ["adjoint"] * 4 + ["grad"])
    spin = rng.choice([0, 0, 0, 2, 2, 2, 1, 3])
    top = 3500 if precision == "fp32" else 2048
    nmaps = 1
    if op == "grad":
        spin, top = rng.choice([0, 2]), 1024
    elif rng.random() < 0.2:
        nmaps, top = rng.choice([2, 3, 5, 16, 40] if precision == "fp32" else [2, 3]), 1024
    lmax = int(round(math.exp(rng.uniform(math.log(96), math.log(top)))))
    mmax = lmax if op == "grad" or rng.random() < 0.7 else rng.randint(lmax // 2, lmax)
    if op == "grad" or rng.random() < 0.6:
        nside, npoints = max(32, lmax // 2 - rng.randint(0, 9)), 0
    else:
        nside, npoints = 0, int(round(math.exp(rng.uniform(math.log(20000), math.log(3 * lmax * lmax + 30000)))))
    c = _case("", op, spin, lmax, precision, epsilon, nside=nside, npoints=npoints, mmax=mmax, nmaps=nmaps)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------ inputs
def _ncomp(case):
    return 1 if case["spin"] == 0 else 2


def _npoints(case):
    return 12 * case["nside"] ** 2 if case["nside"] else case["npoints"]


def _nalm(case):
    return (case["mmax"] + 1) * (2 * case["lmax"] + 2 - case["mmax"]) // 2


def _centres(n, dev):
    """theta, phi of the ring centres of a HEALPix grid (Gorski et al. 2005), ring order."""
    i = np.arange(1, 4 * n)
    cap = np.minimum(i, 4 * n - i)
    polar = cap < n
    z = np.where(polar, 0.0, 4.0 / 3.0 - 2.0 * i / (3.0 * n))
    th = np.where(polar, 2.0 * np.arcsin(np.minimum(1.0, cap / (math.sqrt(6.0) * n))), np.arccos(z))
    th = np.where(polar & (i > 2 * n), math.pi - th, th)
    npix = np.where(polar, 4 * cap, 4 * n)
    shift = np.where(polar, 0.5, 1.0 - 0.5 * ((i - n + 1) % 2))
    start = np.concatenate([[0], np.cumsum(npix)[:-1]])
    cnt = torch.as_tensor(npix, device=dev)
    th, off, st, np_ = (torch.repeat_interleave(torch.as_tensor(v, dtype=torch.float64, device=dev), cnt)
                        for v in (th, shift, start, npix))
    k = torch.arange(int(npix.sum()), dtype=torch.float64, device=dev)
    return th, (k - st + off) * (2.0 * math.pi) / np_


def _points(case, gen, dev, displace=True):
    if not case["nside"]:
        u = torch.rand(3, case["npoints"], dtype=torch.float64, device=dev, generator=gen)
        return torch.acos(2.0 * u[0] - 1.0), 2.0 * math.pi * u[1], math.pi * (2.0 * u[2] - 1.0)
    th, ph = _centres(case["nside"], dev)
    if not displace:
        return th, ph, None
    sig = 2.5 * ARCMIN / math.sqrt(2.0)
    d = sig * torch.randn(3, th.numel(), dtype=torch.float64, device=dev, generator=gen)
    sin = torch.clamp(torch.sin(th), min=1e-3)
    chi = torch.clamp(d[2] * torch.cos(th) / sin, -math.pi, math.pi)
    t2, p2 = th + d[0], ph + d[1] / sin
    over = t2.abs() > math.pi
    p2 = torch.where(over | (t2 < 0), p2 + math.pi, p2)
    t2 = t2.abs()
    t2 = torch.where(over, 2.0 * math.pi - t2, t2)
    return t2, torch.remainder(p2, 2.0 * math.pi), chi


def _lm(lmax, mmax, dev):
    m = torch.repeat_interleave(torch.arange(mmax + 1, device=dev), torch.arange(lmax + 1, lmax - mmax, -1, device=dev))
    base = m * (2 * lmax + 1 - m) // 2
    return torch.arange(m.numel(), device=dev) - base, m


def _alm(cl, lmax, mmax, lmin, lead, gen, dev):
    """Gaussian a_lm: m = 0 real with variance C_l, m > 0 complex with C_l / 2 per part."""
    ell, m = _lm(lmax, mmax, dev)
    sd = torch.sqrt(cl)[ell] * (ell >= lmin)
    z = torch.randn(*lead, ell.numel(), 2, dtype=torch.float64, device=dev, generator=gen)
    re = torch.where(m == 0, z[..., 0], z[..., 0] * math.sqrt(0.5)) * sd
    im = torch.where(m == 0, torch.zeros_like(z[..., 1]), z[..., 1] * math.sqrt(0.5)) * sd
    return torch.complex(re, im)


def _field(case, gen, dev):
    ell = torch.arange(case["lmax"] + 1, dtype=torch.float64, device=dev)
    cl = (ell + 10.0) ** -2 * torch.exp(-(ell / (0.73 * case["lmax"])) ** 2)
    lead = (_ncomp(case),) if case["nmaps"] == 1 else (case["nmaps"], _ncomp(case))
    return _alm(cl, case["lmax"], case["mmax"], case["spin"], lead, gen, dev)


def _potential(lmax, gen, dev):
    ell = torch.arange(lmax + 1, dtype=torch.float64, device=dev)
    cl = (ell + 1.0) ** -4
    cl[:2] = 0.0
    cl *= (2.5 * ARCMIN) ** 2 / torch.sum((2 * ell + 1) / (4 * math.pi) * ell * (ell + 1) * cl)
    return _alm(cl, lmax, lmax, 2, (), gen, dev)


def _inputs(case, seed, dev):
    """Points, a_lm and map of a forward / adjoint case, in the plan's precision."""
    gen = torch.Generator(device=dev).manual_seed(seed)
    f32 = case["precision"] == "fp32"
    pts = _points(case, gen, dev)
    if case["op"] == "forward":
        return pts, _field(case, gen, dev).to(torch.complex64 if f32 else torch.complex128)
    lead = (_ncomp(case),) if case["nmaps"] == 1 else (case["nmaps"], _ncomp(case))
    return pts, torch.randn(*lead, _npoints(case), dtype=torch.float64, device=dev,
                            generator=gen).to(torch.float32 if f32 else torch.float64)


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    if case["op"] == "grad":
        gen = torch.Generator(device=dev).manual_seed(seed)
        f32 = case["precision"] == "fp32"
        th, ph, _ = _points(case, gen, dev, displace=False)
        model = LensingModel(case["lmax"], th, ph, spin=case["spin"], epsilon=case["epsilon"],
                             precision=case["precision"], device=dev)
        pot = _potential(case["lmax"], gen, dev).requires_grad_()
        x = _field(case, gen, dev).to(torch.complex64 if f32 else torch.complex128).requires_grad_()
        g = torch.randn(_ncomp(case), _npoints(case), dtype=torch.float32 if f32 else torch.float64, device=dev,
                        generator=gen)
        model.set_phi(pot)
        return {"case": case, "model": model, "x": x, "pot": pot, "g": g}
    (th, ph, chi), x = _inputs(case, seed, dev)
    plan = LensPlan(case["lmax"], th, ph, chi if case["spin"] else None, spin=case["spin"], mmax=case["mmax"],
                    epsilon=case["epsilon"], precision=case["precision"], device=dev)
    return {"case": case, "plan": plan, "x": x}


def run(state):
    op = state["case"]["op"]
    if op == "forward":
        return state["plan"].synthesis(state["x"])
    if op == "adjoint":
        return state["plan"].adjoint(state["x"])
    d = lensed(state["model"], state["x"], state["pot"])
    gx, gp = torch.autograd.grad(d, (state["x"], state["pot"]), state["g"])
    return {"map": d.detach(), "grad_x": gx, "grad_phi": gp}


def work(case):
    """Inputs and outputs once; Legendre sums over the (l, m, ring pair) triples that are not negligible
    (about 2/pi of all), two length-L transforms of a 2L x L torus half, 8 x 8 kernel taps a point."""
    esz = 4 if case["precision"] == "fp32" else 8
    nc, n, nalm, lmax = _ncomp(case), _npoints(case), _nalm(case), case["lmax"]
    spins = [case["spin"]]
    passes = case["nmaps"]
    if case["op"] == "grad":  # forward, its adjoint, and the raised / lowered fields with the deflection's adjoint
        spins = [case["spin"]] * 2 + [case["spin"] + 1, max(case["spin"] - 1, 1), 1]
    flops = 0.0
    for s in spins:
        c = 1 if s == 0 else 2
        leg = (2 / math.pi) * nalm * (lmax / 2) * (8 if s == 0 else 24)
        fft = 2 * 5 * c * lmax * (case["mmax"] + 1) * 2 * math.log2(2 * lmax)
        flops += passes * (leg + fft + 2 * 64 * c * n)
    nbytes = esz * (passes * (2 * nc * nalm + nc * n) + (2 if case["spin"] == 0 else 3) * n)
    if case["op"] == "grad":
        nbytes += esz * (2 * nc * nalm + nc * n) + 2 * 16 * nalm
    return {"bytes": float(nbytes), "flops": float(flops)}


# ------------------------------------------------------------------------------------ 64-bit results
def _start_norms(mmax, spin, sigma):
    """sign and norm of the start values at l0 = max(m, spin), relative to their powers of sin and cos."""
    out = []
    for m in range(mmax + 1):
        if m >= spin:
            v = math.comb(2 * m, m + sigma) / 4 ** m
            out.append((-1) ** m * math.sqrt((2 * m + 1) / (4 * math.pi) * v))
        else:
            v = math.comb(2 * spin, spin + m) * (2 * spin + 1) / (4 * math.pi)
            out.append((-1) ** (m if sigma > 0 else spin) * math.sqrt(v))
    return out


class _Lambda:
    """s lambda_lm at the given colatitudes for all m at once, degree by degree (plain three-term recursion;
    below lmax ~1900 its smallest relevant start values stay inside the double range)."""

    def __init__(self, case, sigma, theta):
        self.mmax, self.spin, self.sigma = case["mmax"], case["spin"], sigma
        dev = theta.device
        self.m = torch.arange(self.mmax + 1, dtype=torch.float64, device=dev)
        self.x = torch.cos(theta)
        self.sin, self.s2, self.c2 = torch.sin(theta), torch.sin(theta / 2), torch.cos(theta / 2)
        self.norm = _start_norms(self.mmax, self.spin, sigma)
        self.cur = torch.zeros(self.mmax + 1, theta.numel(), dtype=torch.float64, device=dev)
        self.prev = torch.zeros_like(self.cur)

    def _start(self, m):
        if m >= self.spin:
            v = self.sin ** m * (self.s2 / self.c2) ** self.sigma
        else:
            up = self.spin - m if self.sigma > 0 else self.spin + m
            v = self.c2 ** up * self.s2 ** (2 * self.spin - up)
        return self.norm[m] * v

    def at(self, l):
        """Values of degree l for m = 0..min(l, mmax) (degrees in order from the spin upwards)."""
        s, top = self.spin, min(l, self.mmax) + 1
        if l == s:
            for m in range(top):
                self.cur[m] = self._start(m)
            return self.cur[:top]
        old = min(l - 1, self.mmax) + 1
        m = self.m[:old]

        def k(q):
            return torch.sqrt((q * q - m * m) * (q * q - s * s) / (q * q * (4.0 * q * q - 1.0)))

        a1 = k(float(l))
        a0 = k(float(l - 1)) if l > 1 else torch.zeros_like(m)
        p, c = self.prev[:old], self.cur[:old]
        p.mul_(-(a0 / a1)[:, None])
        p.addcmul_(c / a1[:, None], self.x[None, :])
        if s:
            p.addcmul_(c, (m * (self.sigma / (l * (l - 1.0))) / a1)[:, None])
        self.prev, self.cur = self.cur, self.prev
        if old < top:
            self.cur[l] = self._start(l)
            self.prev[l] = 0.0
        return self.cur[:top]


def _chunks(n, mmax):
    step = max(1, int(1.2e8 / (mmax + 1)))
    return [slice(a, min(n, a + step)) for a in range(0, n, step)]


def _exact_forward(case, pts, alm):
    lmax, mmax, s = case["lmax"], case["mmax"], case["spin"]
    theta, phi, chi = pts
    a = alm.to(torch.complex128).reshape(_ncomp(case), -1)
    base = [m * (2 * lmax + 1 - m) // 2 for m in range(mmax + 1)]
    out = torch.empty(_ncomp(case), theta.numel(), dtype=torch.float64, device=theta.device)
    idx0 = torch.as_tensor(base, device=theta.device)
    m = torch.arange(mmax + 1, dtype=torch.float64, device=theta.device)
    for c in _chunks(theta.numel(), mmax):
        gens = [_Lambda(case, sg, theta[c]) for sg in ((0,) if s == 0 else (s, -s))]
        acc = [[torch.zeros_like(g.cur), torch.zeros_like(g.cur)] for g in gens]
        for l in range(s, lmax + 1):
            top = min(l, mmax) + 1
            v = a[:, idx0[:top] + l]
            k = [v[0]] if s == 0 else [v[0] + 1j * v[1], v[0].conj() + 1j * v[1].conj()]
            for g, z, ac in zip(gens, k, acc):
                lam = g.at(l)
                ac[0][:top].addcmul_(lam, z.real[:, None])
                ac[1][:top].addcmul_(lam, z.imag[:, None])
        ang = m[:, None] * phi[c][None, :]
        co, si = torch.cos(ang), torch.sin(ang)
        if s == 0:
            w = torch.where(m == 0, 1.0, 2.0)[:, None]
            out[0, c] = torch.sum(w * (acc[0][0] * co - acc[0][1] * si), 0)
            continue
        q = (m > 0).to(torch.float64)[:, None] * (-1) ** s
        re = -torch.sum(acc[0][0] * co - acc[0][1] * si + q * (acc[1][0] * co + acc[1][1] * si), 0)
        im = -torch.sum(acc[0][1] * co + acc[0][0] * si + q * (acc[1][1] * co - acc[1][0] * si), 0)
        cx, sx = torch.cos(s * chi[c]), torch.sin(s * chi[c])
        out[0, c], out[1, c] = re * cx - im * sx, re * sx + im * cx
    return out


def _exact_adjoint(case, pts, x):
    lmax, mmax, s = case["lmax"], case["mmax"], case["spin"]
    theta, phi, chi = pts
    x = x.to(torch.float64).reshape(_ncomp(case), -1)
    idx0 = torch.as_tensor([m * (2 * lmax + 1 - m) // 2 for m in range(mmax + 1)], device=theta.device)
    out = torch.zeros(_ncomp(case), _nalm(case), dtype=torch.complex128, device=theta.device)
    m = torch.arange(mmax + 1, dtype=torch.float64, device=theta.device)
    for c in _chunks(theta.numel(), mmax):
        ang = m[:, None] * phi[c][None, :]
        co, si = torch.cos(ang), torch.sin(ang)
        if s == 0:
            zs = [(x[0, c] * co, -x[0, c] * si)]
        else:  # e^{-is chi} (Q + iU) e^{-im phi}  and  e^{+is chi} (Q - iU) e^{-im phi}
            cx, sx = torch.cos(s * chi[c]), torch.sin(s * chi[c])
            re, im = x[0, c] * cx + x[1, c] * sx, x[1, c] * cx - x[0, c] * sx
            zs = [(re * co + im * si, im * co - re * si), (re * co - im * si, -im * co - re * si)]
        gens = [_Lambda(case, sg, theta[c]) for sg in ((0,) if s == 0 else (s, -s))]
        for l in range(s, lmax + 1):
            top = min(l, mmax) + 1
            u = []
            for g, (zr, zi) in zip(gens, zs):
                lam = g.at(l)
                u.append(torch.complex(torch.einsum("mp,mp->m", lam, zr[:top]), torch.einsum("mp,mp->m", lam, zi[:top])))
            at = idx0[:top] + l
            if s == 0:
                out[0, at] += u[0]
            else:
                v = (-1) ** s * u[1]
                out[0, at] += -0.5 * (u[0] + v)
                out[1, at] += 0.5j * (u[0] - v)
    return out


def exact(case, seed):
    cost = case["nmaps"] * _npoints(case) * _nalm(case) * (1 if case["spin"] == 0 else 3)
    if cost > 4e11 or case["lmax"] > 1800 or case["op"] == "grad":
        return None
    dev = torch.device("cuda", torch.cuda.current_device())
    pts, x = _inputs(case, seed, dev)
    one = _exact_forward if case["op"] == "forward" else _exact_adjoint
    if case["nmaps"] == 1:
        return one(case, pts, x)
    return torch.stack([one(case, pts, v) for v in x])
