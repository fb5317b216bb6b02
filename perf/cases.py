"""Timed cases of the mass-mapping operators and solvers, each one pass through the public API.

The cases stand for what a user of the library runs: single operator applications (the spin-2
synthesis that simulates shear, the weighted transpose that forms the right-hand side, and H, the
operator every CG iteration applies) in both precisions, from the smallest plan of the tests to
the largest one of the benchmark, on full skies, caps and DES-like footprints, for one and for
several right-hand sides; the batched operator over uneven instances; the flat-sky operator; and
whole calls: a mixed-precision solve and a differentiated solve.

Inputs are seeded and drawn on the device: κ_E a Gaussian field with C_l = 1e-4 (l + 10)^-2 and a
weaker κ_B, galaxy counts Poisson on the footprint, N^-1 = counts / σ_e^2, shape noise of that
variance.  Solves run to a relative residual of 1e-12, so that the solution is determined to
FP64 comparison accuracy and does not depend on the path the iterations took.  FP32 operators
are listed up to lmax 2048 (1024 on noise-dominated maps): their rounding error grows with lmax.
"""
import math

import numpy as np
import torch

from paper_2606_06175_gb300 import akra as A
from paper_2606_06175_gb300.autograd import akra_solve

SIGMA_E = 0.26
LAMBDA = 1e-3
TOL = 1e-12
MAXITER = 4000
PREC = {"f32": A.F32, "f64": A.F64, "mixed": A.MIXED}
BATCH_SHAPE = (1.0, 0.5, 0.25)   # nside of the batch's instances relative to the largest


def listed():
    return [
        # smallest plan of the tests (30-degree cap, Nside 32): launches and latency count
        dict(name="h64_cap32", op="h", prec="f64", nside=32, lmax=64, rhs=1, sky="cap"),
        # small simulation on a grid that is no power of two, odd band limit
        dict(name="synth32_full96", op="synth", prec="f32", nside=96, lmax=251, rhs=3, sky="full"),
        # simulating the shear of a full sky in double precision
        dict(name="synth64_full384", op="synth", prec="f64", nside=384, lmax=768, rhs=1, sky="full"),
        # right-hand side of a noisy survey: the weighted transpose
        dict(name="at32_des1024", op="at", prec="f32", nside=1024, lmax=1024, rhs=1, sky="des"),
        # one FP32 H: the inner CG iteration at the Nside 512 workload
        dict(name="h32_des512", op="h", prec="f32", nside=512, lmax=1024, rhs=1, sky="des"),
        # one FP32 H at the benchmark's Nside, band limit 2048
        dict(name="h32_des2048", op="h", prec="f32", nside=2048, lmax=2048, rhs=1, sky="des"),
        # noise realisations: H of several right-hand sides, tensor-core synthesis as the tuner picks
        dict(name="h32_des1024_rhs8", op="h", prec="f32", nside=1024, lmax=2048, rhs=8, sky="des", tc=8),
        # outer residual of the refinement at the benchmark's full size
        dict(name="h64_des2048", op="h", prec="f64", nside=2048, lmax=4096, rhs=1, sky="des"),
        # uneven instances in one batched pass (the batched inner iteration)
        dict(name="batch32_512_256_128", op="batch", prec="f32", nside=512, lmax=1024, rhs=4, sky="des"),
        # flat-sky survey patch
        dict(name="flat32_2048", op="flat", prec="f32", nside=2048, lmax=0, rhs=1, sky="patch"),
        # a whole reconstruction
        dict(name="solve_mixed_des256", op="solve", prec="mixed", nside=256, lmax=512, rhs=1, sky="des"),
        # loss gradient through a reconstruction (forward and backward)
        dict(name="grad_mixed_des128", op="grad", prec="mixed", nside=128, lmax=256, rhs=1, sky="des"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["synth", "at", "h", "h", "h", "h", "batch", "flat", "solve", "grad"])
    sky = rng.choice(["des", "des", "full", "cap"])
    if op == "flat":
        n = 2 ** rng.randint(6, 12)
        return dict(op="flat", prec=rng.choice(["f32", "f32", "f64"]) if n <= 2048 else "f32", nside=n, lmax=0,
                    rhs=rng.choice([1, 1, 2, 3]) if n <= 2048 else 1, sky="patch")
    if op in ("solve", "grad"):
        n = _log_int(rng, 24, 200)
        return dict(op=op, prec="mixed" if n > 64 else rng.choice(["mixed", "f64"]), nside=n,
                    lmax=_log_int(rng, n, 2 * n), rhs=rng.choice([1, 1, 2]), sky=rng.choice(["des", "cap"]))
    if op == "batch":
        n = 4 * _log_int(rng, 16, 150)
        return dict(op="batch", prec="f32", nside=n, lmax=_log_int(rng, n, 2 * n), rhs=rng.randint(1, 6), sky="des")
    prec = rng.choice(["f32", "f32", "f64"])
    n = _log_int(rng, 24, 2048 if prec == "f32" else 1024)
    top = 1024 if op == "at" and prec == "f32" else 2048
    lmax = min(top, _log_int(rng, n, 2 * n))
    rhs = rng.choice([1, 1, 1, 2, 3, 5]) if n <= 600 else 1
    return dict(op=op, prec=prec, nside=n, lmax=lmax, rhs=rhs, sky=sky)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _rings(nside):
    """z, pixels, first pixel and azimuth of the first pixel of every HEALPix ring."""
    i = np.arange(1, 4 * nside)
    k = np.minimum(i, 4 * nside - i)
    polar = k < nside
    z = np.where(polar, 1 - k * k / (3.0 * nside * nside), 4.0 / 3 - 2 * k / (3.0 * nside))
    n = np.where(polar, 4 * k, 4 * nside)
    shift = np.where(polar, 1, (k - nside + 1) % 2)
    return np.where(i <= 2 * nside, z, -z), n, np.cumsum(n) - n, math.pi * shift / n


def _pixels(nside, dev):
    z, n, first, phi0 = (torch.from_numpy(np.ascontiguousarray(v)).to(dev) for v in _rings(nside))
    ring = torch.repeat_interleave(torch.arange(len(z), device=dev), n)
    j = torch.arange(12 * nside * nside, device=dev) - first[ring]
    return z[ring], phi0[ring] + 2 * math.pi * j / n[ring]


def _footprint(sky, nside, gen, dev):
    z, phi = _pixels(nside, dev)
    if sky == "full":
        return torch.ones_like(z, dtype=torch.bool)
    if sky == "cap":   # 30 degrees around dec -50, RA 30
        d, r = math.radians(-50.0), math.radians(30.0)
        dot = (1 - z * z).clamp(min=0).sqrt() * torch.cos(phi - r) * math.cos(d) + z * math.sin(d)
        return dot >= math.cos(math.radians(30.0))
    # DES-like: a band in declination plus an equatorial strip, edges displaced by up to a degree
    ph = 2 * math.pi * torch.rand(4, device=dev, dtype=torch.float64, generator=gen)
    dec, ra = torch.rad2deg(torch.asin(z)), torch.rad2deg(phi)
    band = (dec >= -60 + torch.sin(3 * phi + ph[0])) & (dec <= -40 + torch.sin(5 * phi + ph[1])) & (ra < 295.1)
    strip = (dec > -41) & (dec <= torch.sin(4 * phi + ph[2])) & (ra <= 10 + torch.sin(8 * z + ph[3]))
    return band | strip


def _ninv(sky, nside, gen, dev):
    fp = _footprint(sky, nside, gen, dev)
    nbar = 5.6 * 4 * math.pi / (12 * nside * nside) * (180 * 60 / math.pi) ** 2
    counts = torch.poisson(torch.full(fp.shape, nbar, device=dev, dtype=torch.float64), generator=gen)
    return torch.where(fp, counts / SIGMA_E ** 2, torch.zeros_like(counts))


def _lm(lmax, dev):
    m = torch.repeat_interleave(torch.arange(lmax + 1, device=dev), torch.arange(lmax + 1, 0, -1, device=dev))
    return torch.arange((lmax + 1) * (lmax + 2) // 2, device=dev) - (m * (2 * lmax + 1 - m)) // 2, m


def _kappa(lmax, rhs, gen, dev):
    """[rhs, 2, ntri] complex128 (κ_E, κ_B)."""
    l, m = _lm(lmax, dev)
    amp = 1e-2 / (l + 10.0)
    amp[l < 2] = 0
    x = torch.randn((rhs, 2, len(l), 2), device=dev, dtype=torch.float64, generator=gen)
    x *= torch.where(m == 0, amp, amp / math.sqrt(2))[:, None]
    x[:, 1] *= 0.1
    x[:, :, m == 0, 1] = 0
    return torch.view_as_complex(x)


def _noise(ninv, rhs, gen):
    sd = torch.where(ninv > 0, ninv, torch.ones_like(ninv)).rsqrt() * (ninv > 0)
    return torch.randn((rhs, 2, ninv.numel()), device=ninv.device, dtype=torch.float64, generator=gen) * sd


def _shear(plan, ninv, kappa, gen):
    y = A.akra_apply_A(plan, A.F64, kappa) + _noise(ninv, kappa.shape[0], gen)
    return y * (ninv > 0)


def _flat_inputs(n, rhs, gen, dev):
    """Weights of a rectangular patch over 70 % x 50 % of the grid, and the transform of κ."""
    c = torch.arange(n, device=dev, dtype=torch.float64) / n
    ph = 2 * math.pi * torch.rand(2, device=dev, dtype=torch.float64, generator=gen)
    e0, e1 = 0.02 * torch.sin(6 * math.pi * c + ph[0]), 0.02 * torch.sin(8 * math.pi * c + ph[1])
    fp = ((c[None, :] - 0.5).abs() < 0.35 + e0[:, None]) & ((c[:, None] - 0.5).abs() < 0.25 + e1[None, :])
    counts = torch.poisson(torch.full((n, n), 5.6 * 0.86 ** 2, device=dev, dtype=torch.float64), generator=gen)
    ninv = torch.where(fp, counts / SIGMA_E ** 2, torch.zeros_like(counts)).reshape(-1)
    k = torch.fft.fftfreq(n, 1.0 / n, device=dev, dtype=torch.float64)
    amp = 1e-2 / ((k[None, :] ** 2 + k[:, None] ** 2).sqrt() + 10)
    x = amp * torch.fft.fft2(torch.randn((rhs, n, n), device=dev, dtype=torch.float64, generator=gen), norm="ortho")
    x[:, 0, 0] = 0
    return ninv, x


def _instances(case):
    return [(max(4, int(case["nside"] * f)), max(4, int(case["lmax"] * f))) for f in BATCH_SHAPE]


def _inputs(case, seed):
    """Everything that is drawn: the same for the timed call and for its value in 64 bits.  FP32
    cases draw values that FP32 holds."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(seed)
    f32 = case["prec"] == "f32"

    def hold(t):
        return t.to(torch.complex64 if t.is_complex() else torch.float32) if f32 else t

    if case["op"] == "flat":
        ninv, x = _flat_inputs(case["nside"], case["rhs"], gen, dev)
        return dict(ninv=ninv, x=hold(x))
    if case["op"] == "batch":
        return dict(parts=[dict(ninv=_ninv(case["sky"], n, gen, dev), x=hold(_kappa(l, case["rhs"], gen, dev)))
                           for n, l in _instances(case)])
    got = dict(x=hold(_kappa(case["lmax"], case["rhs"], gen, dev)))
    if case["op"] != "synth":
        got["ninv"] = _ninv(case["sky"], case["nside"], gen, dev)
    if case["op"] == "at":   # noise-dominated maps, as a survey's are
        got["map"] = hold(_noise(got["ninv"], case["rhs"], gen))
    if case["op"] in ("solve", "grad"):
        got["gen"] = gen
    return got


def prepare(case, seed):
    s = _inputs(case, seed)
    s.update(op=case["op"], prec=PREC[case["prec"]])
    if case["op"] == "flat":
        s["plan"] = A.akra_flat_plan_create(case["nside"])
        A.akra_plan_set_weights(s["plan"], s["ninv"], LAMBDA)
        return s
    if case["op"] == "batch":
        plans = []
        for (n, l), part in zip(_instances(case), s["parts"]):
            plans.append(A.akra_plan_create(n, l))
            A.akra_plan_set_weights(plans[-1], part["ninv"], LAMBDA)
        s["batch"] = A.akra_batch_create(plans, [case["rhs"]] * len(plans))
        return s
    s["plan"] = A.akra_plan_create(case["nside"], case["lmax"])
    if "ninv" in s:
        A.akra_plan_set_weights(s["plan"], s["ninv"], LAMBDA)
    if case.get("tc"):
        A.akra_plan_set_tc_synthesis(s["plan"], case["rhs"], case["tc"])
    if case["op"] in ("solve", "grad"):
        s["y"] = _shear(s["plan"], s["ninv"], s.pop("x"), s.pop("gen"))
    return s


def run(s):
    op, prec = s["op"], s["prec"]
    if op == "synth":
        return A.akra_synth_spin2(s["plan"], prec, s["x"])
    if op == "at":
        return A.akra_apply_At(s["plan"], prec, s["map"], weighted=True)
    if op in ("h", "flat"):
        return A.akra_apply_H(s["plan"], prec, s["x"])
    if op == "batch":
        return A.akra_batch_apply_H(s["batch"], [p["x"] for p in s["parts"]])
    if op == "solve":
        return A.akra_cg_solve(s["plan"], prec, s["y"], tol=TOL, maxiter=MAXITER)[0]
    y, ninv = s["y"].detach().requires_grad_(), s["ninv"].detach().requires_grad_()
    x = akra_solve(y, ninv, s["plan"], prec, tol=TOL, maxiter=MAXITER, lam=LAMBDA)
    x.abs().square().sum().backward()
    return x.detach(), y.grad, ninv.grad


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _transform_work(nside, lmax, rhs, size, rings, sides):
    """`sides` Legendre transforms of the (l, m, ring) triangle, 8 multiply-adds per step with one
    right-hand side, and their ring FFTs."""
    ntri, npix = (lmax + 1) * (lmax + 2) // 2, rings * 3.0 * nside
    flops = sides * (2.0 * (4 + 4 * rhs) * ntri * rings + rhs * 10.0 * npix * math.log2(4 * nside + 1))
    return flops, 4.0 * rhs * ntri * size, 2.0 * rhs * npix * size


def _rings_of(sky, nside):
    return {"full": 4 * nside - 1, "cap": nside, "des": 1.37 * nside}[sky]


def work(case):
    size = 4 if case["prec"] == "f32" else 8
    n, l, r = case["nside"], case["lmax"], case["rhs"]
    if case["op"] == "flat":
        return dict(bytes=float(size * n * n * (4 * r + 1)), flops=r * n * n * (20.0 * math.log2(n) + 20))
    if case["op"] == "batch":
        got = [work(dict(case, op="h", nside=a, lmax=b)) for a, b in _instances(case)]
        return dict(bytes=sum(g["bytes"] for g in got), flops=sum(g["flops"] for g in got))
    rings = _rings_of(case["sky"], n)
    sides = 1 if case["op"] in ("synth", "at") else 2
    flops, alm, maps = _transform_work(n, l, r, size, rings, sides)
    if case["op"] in ("synth", "at"):
        return dict(bytes=alm + maps + (0 if case["op"] == "synth" else 3.0 * n * rings * size), flops=flops)
    if case["op"] == "h":
        return dict(bytes=2 * alm + 3.0 * n * rings * size, flops=flops)
    solves = 1 if case["op"] == "solve" else 2   # a few hundred iterations each
    return dict(bytes=solves * (2 * alm + maps), flops=solves * 300 * flops)


# ---------------------------------------------------------------------------
# values in 64 bits, by plain torch
# ---------------------------------------------------------------------------
class _Sphere:
    """Spin-2 transforms on the listed HEALPix rings by direct recurrence in l over all (m, ring)."""

    def __init__(self, nside, lmax, rows, dev):
        z, n, first, phi0 = _rings(nside)
        self.nside, self.lmax, self.dev = nside, lmax, dev
        self.rows, self.n, self.first = rows, n, first
        self.x = torch.from_numpy(z[rows]).to(dev)
        k = np.minimum(rows + 1, 4 * nside - 1 - rows).astype(np.float64)
        omz = np.where(k < nside, k * k / (3.0 * nside * nside), (2 * k - nside) / (3.0 * nside))   # 1 - |z|
        s2, c2 = 0.5 * omz, 0.5 * (2 - omz)
        north = rows + 1 <= 2 * nside
        self.ls = torch.from_numpy(0.5 * np.log2(np.where(north, s2, c2))).to(dev)   # log2 sin(θ/2)
        self.lc = torch.from_numpy(0.5 * np.log2(np.where(north, c2, s2))).to(dev)
        m = torch.arange(lmax + 1, device=dev, dtype=torch.float64)
        self.m = m
        self.turn = torch.polar(torch.ones(len(rows), lmax + 1, device=dev, dtype=torch.float64),
                                torch.from_numpy(phi0[rows]).to(dev)[:, None] * m[None, :])

    def functions(self):
        """Yields (l, 2λ_lm, -2λ_lm) as [ring, m <= l] for l = 2 .. lmax."""
        L, x, m = self.lmax, self.x[:, None], self.m[None, :]
        mm = torch.clamp(m, min=2)
        a, b = m + 2, (m - 2).abs()
        c = 0.5 * (torch.log2(2 * mm + 1) - math.log2(4 * math.pi) +
                   (torch.lgamma(2 * mm + 1) - torch.lgamma(a + 1) - torch.lgamma(b + 1)) / math.log(2))
        sp = 1 - 2 * (m % 2)
        sm = torch.where(m >= 2, sp, torch.ones_like(sp))
        lp = c + a * self.ls[:, None] + b * self.lc[:, None]
        lm = c + b * self.ls[:, None] + a * self.lc[:, None]
        e = torch.clamp(torch.floor((torch.maximum(lp, lm) + 300) / 600), max=0)   # value = v 2^(600 e)
        seed_p, seed_m = sp * torch.exp2(lp - 600 * e), sm * torch.exp2(lm - 600 * e)
        vp, vm, op, om = (torch.zeros_like(seed_p) for _ in range(4))
        vp[:, :3], vm[:, :3] = seed_p[:, :3], seed_m[:, :3]
        for l in range(2, L + 1):
            if l > 2:
                vp[:, l], vm[:, l] = seed_p[:, l], seed_m[:, l]
            live = (e == 0)[:, :l + 1]
            yield l, vp[:, :l + 1] * live, vm[:, :l + 1] * live
            if l == L:
                return
            q = m[:, :l + 1]
            A_ = math.sqrt((2 * l + 3) / (2 * l + 1)) * (l + 1) * (2 * l + 1) / \
                torch.sqrt(((l + 1.0) ** 2 - q * q) * ((l + 1.0) ** 2 - 4))
            B_ = torch.sqrt((l * l - q * q) * (l * l - 4.0)) / (l * (2 * l + 1)) * math.sqrt((2 * l + 1) / (2 * l - 1))
            s = 2 * A_ * q / (l * (l + 1.0))
            np_ = (A_ * x + s) * vp[:, :l + 1] - A_ * B_ * op[:, :l + 1]
            nm_ = (A_ * x - s) * vm[:, :l + 1] - A_ * B_ * om[:, :l + 1]
            op[:, :l + 1], om[:, :l + 1], vp[:, :l + 1], vm[:, :l + 1] = vp[:, :l + 1], vm[:, :l + 1], np_, nm_
            if l % 16 == 0:
                big = (e < 0) & (torch.maximum(vp.abs(), vm.abs()) > 2.0 ** 300)
                f = torch.exp2(-600.0 * big.double())
                vp, vm, op, om, e = vp * f, vm * f, op * f, om * f, e + big

    def _column(self, l):
        m = torch.arange(l + 1, device=self.dev)
        return (m * (2 * self.lmax + 1 - m)) // 2 + l

    def _ks(self, l, ks):
        return -math.sqrt((l - 1.0) * (l + 2.0) / (l * (l + 1.0))) if ks else -1.0

    def _groups(self):
        for n in np.unique(self.n[self.rows]):
            at = np.nonzero(self.n[self.rows] == n)[0]
            px = torch.from_numpy(self.first[self.rows[at]][:, None] + np.arange(n)[None, :]).to(self.dev)
            yield int(n), torch.from_numpy(at).to(self.dev), px

    def synth(self, alm, ks):
        """[R, 2, ntri] -> [R, npix] complex γ1 + iγ2 (zero off the rings)."""
        R, K, L = alm.shape[0], len(self.rows), self.lmax
        fp = torch.zeros((R, K, L + 1), device=self.dev, dtype=torch.complex128)
        fm = torch.zeros_like(fp)
        for l, p, q in self.functions():
            col = alm[:, :, self._column(l)] * self._ks(l, ks)
            col[:, :, 0] = col[:, :, 0].real.to(col.dtype)
            c, d = col[:, 0] + 1j * col[:, 1], col[:, 0] - 1j * col[:, 1]
            fp[:, :, :l + 1] += c[:, None] * p
            fm[:, :, :l + 1] += d[:, None] * q
        fp, fm = fp * self.turn, (fm * self.turn).conj()
        out = torch.zeros((R, 12 * self.nside ** 2), device=self.dev, dtype=torch.complex128)
        m = torch.arange(L + 1, device=self.dev)
        for n, at, px in self._groups():
            bins = torch.zeros((R, len(at), n), device=self.dev, dtype=torch.complex128)
            bins.index_add_(2, m % n, fp[:, at])
            bins.index_add_(2, (-m[1:]) % n, fm[:, at, 1:])
            out[:, px] = torch.fft.ifft(bins, dim=2) * n
        return out

    def adjoint(self, u, ks):
        """[R, npix] complex -> [R, 2, ntri]: the transpose of synth in the real inner product."""
        R, K, L = u.shape[0], len(self.rows), self.lmax
        m = torch.arange(L + 1, device=self.dev)
        gp = torch.zeros((R, K, L + 1), device=self.dev, dtype=torch.complex128)
        gm = torch.zeros_like(gp)
        for n, at, px in self._groups():
            f = torch.fft.fft(u[:, px], dim=2)
            gp[:, at], gm[:, at] = f[:, :, m % n], f[:, :, (-m) % n]
        gp, gm = gp * self.turn.conj(), gm.conj() * self.turn.conj()
        out = torch.zeros((R, 2, (L + 1) * (L + 2) // 2), device=self.dev, dtype=torch.complex128)
        for l, p, q in self.functions():
            a, b = (gp[:, :, :l + 1] * p).sum(1), (gm[:, :, :l + 1] * q).sum(1)
            f, at = 0.5 * self._ks(l, ks), self._column(l)
            out[:, 0, at], out[:, 1, at] = f * (a + b), -1j * f * (a - b)
        out[:, :, :L + 1] = out[:, :, :L + 1].real.to(out.dtype)
        return out


def _weights(nside, ninv):
    omega = 4 * math.pi / (12.0 * nside * nside)
    on = ninv > 0
    lam = LAMBDA * float(ninv.sum()) / max(1, int(on.sum()))
    _, n, first, _ = _rings(nside)
    ring = torch.repeat_interleave(torch.arange(len(n), device=ninv.device), torch.from_numpy(n).to(ninv.device))
    rows = np.nonzero(torch.bincount(ring, weights=on.double(), minlength=len(n)).cpu().numpy() > 0)[0]
    return omega * ninv, lam, rows


def _exact_h(nside, lmax, ninv, x):
    w, lam, rows = _weights(nside, ninv)
    sphere = _Sphere(nside, lmax, rows, x.device)
    y = sphere.adjoint(sphere.synth(x, True) * w, True) + lam * x
    y[:, :, :lmax + 1] = y[:, :, :lmax + 1].real.to(y.dtype)
    return y


def exact(case, seed):
    op, n, l = case["op"], case["nside"], case["lmax"]
    if op in ("solve", "grad"):
        return None
    if op != "flat" and (case["sky"] == "full" and n > 700 or l > 2048 or n * case["rhs"] > 4096):
        return None   # tens of seconds
    s = _inputs(case, seed)
    if op == "batch":
        return [_exact_h(a, b, p["ninv"], p["x"].to(torch.complex128)) for (a, b), p in zip(_instances(case), s["parts"])]
    x = s["x"].to(torch.complex128)
    if op == "flat":
        k = torch.fft.fftfreq(n, 1.0 / n, device=x.device, dtype=torch.float64)
        k1, k2 = k[None, :], k[:, None]
        kk = k1 ** 2 + k2 ** 2
        D = torch.where(kk > 0, (k1 ** 2 - k2 ** 2 + 2j * k1 * k2) / kk.clamp(min=1), 0j)
        on = s["ninv"] > 0
        lam = LAMBDA * float(s["ninv"].sum()) / max(1, int(on.sum()))
        g = torch.fft.ifft2(D * x, norm="ortho") * s["ninv"].reshape(n, n)
        return D.conj() * torch.fft.fft2(g, norm="ortho") + lam * x
    if op == "h":
        return _exact_h(n, l, s["ninv"], x)
    if op == "at":
        w, _, rows = _weights(n, s["ninv"])
        u = s["map"].double()
        return _Sphere(n, l, rows, x.device).adjoint(torch.complex(u[:, 0], u[:, 1]) * w, True)
    g = _Sphere(n, l, np.arange(4 * n - 1), x.device).synth(x, False)
    return torch.stack([g.real, g.imag], dim=1)
