"""FP32 ring FFT at every block size against the operators' own bound, tol32(L) = 4 · 2^-24 max(L, 16).
(test_gpu_ringfft32_threads.py names that bound but computes it with numpy's float32 eps, which is 2^-23: twice as wide.)"""
import pytest
import torch

from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float((a.to(b.dtype) - b).norm() / b.norm())


@pytest.mark.parametrize("nside,lmax,R", [(8, 16, 1), (8, 16, 90), (64, 100, 2), (64, 100, 20), (100, 150, 9), (256, 300, 3), (512, 512, 2)])
def test_operators_within_the_bound(nside, lmax, R):
    gen = torch.Generator(device=DEV).manual_seed(nside + R)
    p = A.akra_plan_create(nside, lmax)
    A.akra_plan_set_weights(p, torch.rand(p.npix, device=DEV, generator=gen, dtype=torch.float64) + 0.5, 1e-3)
    x = torch.randn(R, 2, p.ntri, 2, device=DEV, generator=gen)
    x[:, :, :lmax + 1, 1] = 0
    x = torch.view_as_complex(x)
    u = torch.randn(R, 2, p.npix, device=DEV, generator=gen)
    tol = 4 * 2.0 ** -24 * max(lmax, 16)
    for f, v in ((A.akra_synth_spin2, x), (A.akra_adjoint_synth_spin2, u), (A.akra_apply_H, x)):
        wide = v.to(torch.complex128) if v.is_complex() else v.double()
        assert rel(f(p, A.F32, v), f(p, A.F64, wide)) < tol, f.__name__
