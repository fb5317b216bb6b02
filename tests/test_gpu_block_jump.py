"""The FP32 Legendre kernels that advance by 16-step blocks with interpolated transfer polynomials
(csrc/akra_legendre_blk.cuh), at the edges of their tiles: ring counts around a chunk of 256, band limits around
16-step blocks and 128-step tiles, rings north and south, footprints that reach a pole (whose last rings stay
with the difference-form kernels), a pair list that needs both rings of some pairs, and several RHS."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
import synthetic as S
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def tol32(lmax):
    return 4 * 2.0 ** -24 * max(lmax, 16)   # the FP32 operators' bound (as in test_gpu_operators.py)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


SKIES = {
    "south": lambda z: (z < -0.1) & (z > -0.95),
    "north_pole": lambda z: z > 0.2,
    "south_pole_and_equator": lambda z: z < 0.06,       # a few pairs need both rings
    "thin": lambda z: (z < -0.5) & (z > -0.52),         # fewer rings than a warp
}


@pytest.mark.parametrize("sky", SKIES)
@pytest.mark.parametrize("N,L", [(64, 128), (64, 159), (100, 257), (128, 130), (150, 300)])
def test_block_jump_H_and_adjoint_match_oracle(sky, N, L):
    rng = np.random.default_rng(1000 * N + L)
    R = 2 if N == 64 else 1
    z = np.cos(O.pixel_angles(N)[0])
    ninv = np.where(SKIES[sky](z), 1.0 + rng.random(12 * N * N), 0.0)
    w = O.Weights(N, ninv, 1e-3)
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
    pairs = [(S.random_alm(L, rng), S.random_alm(L, rng)) for _ in range(R)]
    x = torch.from_numpy(np.stack([np.stack(q) for q in pairs])).to(DEV, torch.complex64)
    y = A.akra_apply_H(p, A.F32, x).cpu().numpy()
    u = rng.normal(size=(R, 2, 12 * N * N)).astype(np.float32)
    b = A.akra_apply_At(p, A.F32, torch.from_numpy(u).to(DEV), weighted=True).cpu().numpy()
    for r in range(R):
        xe, xb = (x[r, f].cpu().numpy().astype(np.complex128) for f in (0, 1))
        assert rel(y[r], np.stack(O.apply_H(N, L, w, xe, xb))) < tol32(L), ("H", sky, r)
        un = u[r].astype(np.float64)
        assert rel(b[r], np.stack(O.rhs_b(N, L, w, un[0], un[1]))) < tol32(L), ("At", sky, r)


def test_block_jump_propagates_non_finite_values():
    """A NaN or infinite coefficient reaches H's result, as in the direct kernels."""
    N, L = 64, 128
    z = np.cos(O.pixel_angles(N)[0])
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, torch.from_numpy(np.where(z < -0.2, 1.0, 0.0)).to(DEV), 1e-3)
    x = torch.ones(p.alm_shape(1), dtype=torch.complex64, device=DEV)
    for bad in (float("nan"), float("inf")):
        xx = x.clone()
        xx[0, 0, O.tri_index(L, 3, 100)] = bad
        assert not bool(torch.isfinite(torch.view_as_real(A.akra_apply_H(p, A.F32, xx))).all())
    assert bool((A.akra_apply_H(p, A.F32, torch.zeros_like(x)) == 0).all())


@pytest.mark.parametrize("N,L,R,group", [(64, 128, 1, 4), (64, 128, 9, 8), (100, 257, 3, 8), (64, 127, 3, 8), (64, 128, 9, 16)])
def test_tensor_core_groups_on_one_ring_footprints(N, L, R, group):
    """Groups of 4 and 8 take the block-jump kernel from lmax 128 on, larger ones and smaller lmax do not; a fixed
    shape keeps the group's own kernel."""
    rng = np.random.default_rng(L + R)
    z = np.cos(O.pixel_angles(N)[0])
    ninv = np.where(SKIES["south"](z), 1.0 + rng.random(12 * N * N), 0.0)
    w = O.Weights(N, ninv, 1e-3)
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
    pairs = [(S.random_alm(L, rng), S.random_alm(L, rng)) for _ in range(R)]
    x = torch.from_numpy(np.stack([np.stack(q) for q in pairs])).to(DEV, torch.complex64)
    plain = A.akra_apply_H(p, A.F32, x)
    A.akra_plan_set_tc_synthesis(p, R, group)
    assert A.akra_plan_get_tc_synthesis(p, R) == group
    y = A.akra_apply_H(p, A.F32, x)
    assert torch.equal(y, plain) == (group <= 8 and L >= 128)
    A.akra_plan_set_shape(p, A.F32, R, 1, 1, 1)
    A.akra_plan_set_tc_synthesis(p, R, group)
    fixed = A.akra_apply_H(p, A.F32, x)
    for r in range(R):
        ref = np.stack(O.apply_H(N, L, w, *pairs[r]))
        assert rel(y[r].cpu().numpy(), ref) < tol32(L), ("H", r)
        assert rel(fixed[r].cpu().numpy(), ref) < tol32(L), ("fixed shape", r)


def test_badly_filled_chunks_keep_the_direct_adjoint_for_several_rhs():
    """557 rings in three chunks of 256: from 3 RHS on the direct adjoint takes A^T, one RHS the block jumps."""
    N, L, R = 380, 130, 3
    z = np.cos(O.pixel_angles(N)[0])
    ninv = np.where(SKIES["south"](z), 1.0, 0.0)
    w = O.Weights(N, ninv, 1e-3)
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
    u = np.random.default_rng(8).normal(size=(R, 2, 12 * N * N)).astype(np.float32)
    ud = torch.from_numpy(u).to(DEV)
    b = A.akra_apply_At(p, A.F32, ud, weighted=True).cpu().numpy()
    one = A.akra_apply_At(p, A.F32, ud[:1], weighted=True).cpu().numpy()
    ref = np.stack(O.rhs_b(N, L, w, *u[0].astype(np.float64)))
    assert rel(b[0], ref) < tol32(L) and rel(one[0], ref) < tol32(L)
    for r in range(1, R):
        assert rel(b[r], np.stack(O.rhs_b(N, L, w, *u[r].astype(np.float64)))) < tol32(L)
