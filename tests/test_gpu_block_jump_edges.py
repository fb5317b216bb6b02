"""The FP32 block-jump Legendre kernels where their number formats and chunks are at an edge: ring counts at and beside
whole chunks of 256, spectra that fall steeply inside the 32 steps that share a scale, and rings of very unequal
weight inside the chunk that shares one.

Bounds: the FP32 operators' tol32(L) = 4 · 2^-24 L on the 2-norm, and for the formats no more than 1.5 times the error of the
direct kernels on the same input (both against the FP64 operator)."""
import numpy as np
import pytest
import torch

from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def tol32(lmax):
    return 4 * 2.0 ** -24 * max(lmax, 16)


def rel(a, b):
    return float((a.to(b.dtype) - b).norm() / b.norm())


def _rings(N):
    """Ring index (0-based, north to south) of every pixel."""
    i = np.arange(1, 4 * N)
    return np.repeat(i - 1, 4 * np.minimum(np.minimum(i, 4 * N - i), N))


def _plan(N, L, ninv):
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
    return p


def _alm(L, seed, amp=None):
    """[1, 2, ntri] complex128, unit normal or of the amplitude amp(l)."""
    m = np.repeat(np.arange(L + 1), np.arange(L + 1, 0, -1))
    l = np.concatenate([np.arange(q, L + 1) for q in range(L + 1)])
    g = np.random.default_rng(seed).normal(size=(2, 2, len(l)))
    g[1][:, m == 0] = 0
    x = g[0] + 1j * g[1]
    if amp is not None:
        x *= amp(l)
    return torch.from_numpy(x[None]).to(DEV).to(torch.complex64)


def _direct(p):
    A.akra_plan_set_shape(p, A.F32, 1, 1, 1, 1)
    A.akra_plan_set_adjoint_shape(p, A.F32, 1, 3, 1)


@pytest.mark.parametrize("count", [1, 31, 255, 256, 257, 511, 512, 513])
def test_ring_counts(count):
    N, L = 300, 310
    ring = _rings(N)   # from six rings south of the equator on; the last is 0.4 rad from the pole
    ninv = np.where((ring >= 605) & (ring < 605 + count), 1.0 + np.random.default_rng(count).random(12 * N * N), 0.0)
    p = _plan(N, L, ninv)
    x = _alm(L, count)
    u = torch.randn(1, 2, 12 * N * N, device=DEV, generator=torch.Generator(device=DEV).manual_seed(count))
    y, b = A.akra_apply_H(p, A.F32, x), A.akra_apply_At(p, A.F32, u, weighted=True)
    assert rel(y, A.akra_apply_H(p, A.F64, x.to(torch.complex128))) < tol32(L)
    assert rel(b, A.akra_apply_At(p, A.F64, u.double(), weighted=True)) < tol32(L)
    _direct(p)
    assert not torch.equal(A.akra_apply_At(p, A.F32, u, weighted=True), b)   # the block jumps had run


SPECTRA = {
    "falling": lambda l: 10.0 ** (-8 * (l % 32) / 31.0),        # eight decades over the 32 steps of a scale
    "rising": lambda l: 10.0 ** (-8 * (31 - l % 32) / 31.0),
    "one_l": lambda l: np.where(l == 77, 1e6, 1.0),
    "low_l": lambda l: np.maximum(l, 2.0) ** -4.0,              # steep over the whole range, as low-l power is
}


@pytest.mark.parametrize("spectrum", SPECTRA)
@pytest.mark.parametrize("N,L", [(64, 128), (128, 300)])
def test_steep_spectra(N, L, spectrum):
    ring = _rings(N)
    p = _plan(N, L, np.where((ring >= 2 * N + 5) & (ring < 4 * N - 30), 1.0, 0.0))
    x = _alm(L, L, SPECTRA[spectrum])
    ref = A.akra_apply_H(p, A.F64, x.to(torch.complex128))
    blk = rel(A.akra_apply_H(p, A.F32, x), ref)
    _direct(p)
    direct = rel(A.akra_apply_H(p, A.F32, x), ref)
    assert blk < tol32(L) and blk <= 1.5 * direct, (blk, direct)


@pytest.mark.parametrize("decades", [4, 8])
@pytest.mark.parametrize("N,L", [(64, 128), (128, 300)])
def test_rings_of_unequal_weight(N, L, decades):
    ring = _rings(N)
    rng = np.random.default_rng(N + decades)
    per_ring = 10.0 ** -(decades * rng.random(4 * N))
    p = _plan(N, L, np.where((ring >= 2 * N + 5) & (ring < 4 * N - 30), per_ring[ring], 0.0))
    x = _alm(L, L)
    u = torch.from_numpy(rng.normal(size=(1, 2, 12 * N * N))).to(DEV).float()
    refs = A.akra_apply_H(p, A.F64, x.to(torch.complex128)), A.akra_apply_At(p, A.F64, u.double(), weighted=True)
    blk = rel(A.akra_apply_H(p, A.F32, x), refs[0]), rel(A.akra_apply_At(p, A.F32, u, weighted=True), refs[1])
    _direct(p)
    direct = rel(A.akra_apply_H(p, A.F32, x), refs[0]), rel(A.akra_apply_At(p, A.F32, u, weighted=True), refs[1])
    for e, d in zip(blk, direct):
        assert e < tol32(L) and e <= 1.5 * d, (blk, direct)
