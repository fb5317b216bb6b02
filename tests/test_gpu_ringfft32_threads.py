"""FP32 ring FFT at every block size: the thread count follows the number of rings and right-hand sides, so one
plan meets several of them.  Longest convolutions from 64 (Nside 8) to 4096 (Nside 512), R from one to the
number that takes the smallest block; the map synthesis, its adjoint and H against the FP64 path.

Tolerance: tol32(L) = 4 eps32 L, that of the operator tests."""
import numpy as np
import pytest
import torch

from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(torch.linalg.vector_norm(a.to(b.dtype) - b) / torch.linalg.vector_norm(b))


@pytest.mark.parametrize("nside,lmax,counts", [(8, 16, (1, 5, 90)), (64, 100, (1, 2, 5, 20)), (100, 150, (1, 4, 9)),
                                               (256, 300, (1, 3)), (512, 512, (1, 2))])
def test_block_sizes(nside, lmax, counts):
    gen = torch.Generator(device=DEV).manual_seed(nside)
    npix, ntri = 12 * nside * nside, (lmax + 1) * (lmax + 2) // 2
    p = A.akra_plan_create(nside, lmax)
    w = torch.rand(npix, device=DEV, generator=gen, dtype=torch.float64) + 0.5
    A.akra_plan_set_weights(p, w, 1e-3)
    tol = 4 * float(np.finfo(np.float32).eps) * lmax
    for R in counts:
        x = torch.randn(R, 2, ntri, 2, device=DEV, generator=gen, dtype=torch.float64)
        x[:, :, :lmax + 1, 1] = 0
        x = torch.view_as_complex(x).contiguous()
        u = torch.randn(R, 2, npix, device=DEV, generator=gen, dtype=torch.float64)
        s = A.akra_synth_spin2(p, A.F32, x.to(torch.complex64))
        a = A.akra_adjoint_synth_spin2(p, A.F32, u.float())
        h = A.akra_apply_H(p, A.F32, x.to(torch.complex64))
        assert rel(s, A.akra_synth_spin2(p, A.F64, x)) < tol, ("synth", R)
        assert rel(a, A.akra_adjoint_synth_spin2(p, A.F64, u)) < tol, ("adjoint", R)
        assert rel(h, A.akra_apply_H(p, A.F64, x)) < tol, ("H", R)
