"""Which Legendre kernel the default shapes take on footprints of one hemisphere, by the bits of the result: the
block-jump kernels and each direct shape sum in an order of their own, so a result equals that of a forced shape
only where that shape ran.  Every result also matches the FP64 operator."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def tol32(lmax):
    return 4 * 2.0 ** -24 * max(lmax, 16)   # as in test_gpu_operators.py


def rel(a, b):
    return float((a.to(b.dtype) - b).norm() / b.norm())


ONE_SIDE, TWO_SIDES = (-0.95, -0.1), (-0.95, 0.02)   # cos(theta); the second needs both rings of a few pairs


def _plan(N, L, sky=ONE_SIDE):
    z = np.cos(O.pixel_angles(N)[0])
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, torch.from_numpy(np.where((z > sky[0]) & (z < sky[1]), 2.0, 0.0)).to(DEV), 1e-3)
    return p


# adjoint of (Nside, lmax, R): the direct shape (ring pairs per thread, RHS per block), or None for the block jumps
ROUTES = [
    (64, 128, 2, None, ONE_SIDE),         # one chunk of rings
    (64, 128, 3, (1, 1), ONE_SIDE),       # 94 pairs
    (200, 250, 2, (3, 1), ONE_SIDE),      # 293 pairs
    (300, 349, 4, (4, 1), TWO_SIDES),     # up to lmax 350, 436 pairs
    (300, 350, 4, None, TWO_SIDES),
    (400, 420, 3, (5, 1), ONE_SIDE),      # 586 pairs that fill three chunks badly
    (345, 420, 3, (5, 1), TWO_SIDES),     # 567 rings, 557 pairs, three chunks
    (345, 420, 2, None, TWO_SIDES),
    (120, 360, 3, None, ONE_SIDE),        # one chunk from lmax 350 on
    (400, 420, 1, None, ONE_SIDE),
    (400, 551, 1, (5, 1), ONE_SIDE),      # one right-hand side from Nside · lmax 220000 on
    (300, 600, 4, None, ONE_SIDE),        # 439 pairs in two chunks that are not badly filled
    (600, 500, 1, (4, 1), ONE_SIDE),      # lmax below Nside, four chunks, 878 pairs
    (480, 479, 1, (3, 1), ONE_SIDE),      # 703 pairs: 768 slots in chunks of 384
    (480, 480, 1, None, ONE_SIDE),
]


@pytest.mark.parametrize("N,L,R,shape,sky", ROUTES)
def test_default_adjoint(N, L, R, shape, sky):
    p = _plan(N, L, sky)
    u = torch.randn(R, 2, 12 * N * N, device=DEV, generator=torch.Generator(device=DEV).manual_seed(N + L + R))
    b = A.akra_apply_At(p, A.F32, u, weighted=True)
    assert rel(b, A.akra_apply_At(p, A.F64, u.double(), weighted=True)) < tol32(L)
    for forced in {(5, 1), (4, 1), shape or (2, 1)}:   # pairs per thread set the order of the sums
        A.akra_plan_set_adjoint_shape(p, A.F32, R, *forced)
        same = torch.equal(A.akra_apply_At(p, A.F32, u, weighted=True), b)
        assert same == (forced == shape), (forced, shape)


@pytest.mark.parametrize("N,L,R,direct", [(64, 128, 3, False), (64, 128, 4, True), (64, 128, 5, False), (400, 420, 8, True),
                                          (300, 1090, 4, True), (300, 1110, 4, False)])
def test_default_synthesis(N, L, R, direct):
    """H with the adjoint's shape fixed: its synthesis is that of the forced shape (1, RG) or the block jumps'."""
    p = _plan(N, L)
    x = torch.randn(R, 2, p.ntri, 2, device=DEV, generator=torch.Generator(device=DEV).manual_seed(N + L + R))
    x[:, :, :L + 1, 1] = 0
    x = torch.view_as_complex(x)
    A.akra_plan_set_adjoint_shape(p, A.F32, R, 2, 1)
    y = A.akra_apply_H(p, A.F32, x)
    assert rel(y, A.akra_apply_H(p, A.F64, x.to(torch.complex128))) < tol32(L)
    A.akra_plan_set_shape(p, A.F32, R, 1, 1, 4 if R >= 4 else 2)
    A.akra_plan_set_adjoint_shape(p, A.F32, R, 2, 1)
    assert torch.equal(A.akra_apply_H(p, A.F32, x), y) == direct


def test_footprint_does_not_change_the_full_sky_shape():
    """The unweighted adjoint over all rings of a plan whose footprint keeps a direct shape of its own."""
    N, L, R = 400, 420, 4
    p = _plan(N, L)
    u = torch.randn(R, 2, 12 * N * N, device=DEV, generator=torch.Generator(device=DEV).manual_seed(1))
    b = A.akra_adjoint_synth_spin2(p, A.F32, u)
    A.akra_plan_set_adjoint_shape(p, A.F32, R, 2, 2)
    assert torch.equal(A.akra_adjoint_synth_spin2(p, A.F32, u), b)
    A.akra_plan_set_adjoint_shape(p, A.F32, R, 5, 1)
    assert not torch.equal(A.akra_adjoint_synth_spin2(p, A.F32, u), b)
