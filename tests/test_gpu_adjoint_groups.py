"""FP32 adjoint of many right-hand sides on a footprint of one hemisphere: the partial sums of the block-jump
kernel's chunks are formed for some right-hand sides at a time where all of them would take more memory than
the direct kernel's and than 4 GB.  Results are those of the right-hand sides by themselves, to the bit."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def test_groups_give_the_single_results_and_bound_the_partial_sums():
    N, L, R = 1024, 2048, 33
    z = np.cos(O.pixel_angles(N)[0])
    ninv = torch.from_numpy(np.where((z > -0.86) & (z < 0.0), 2.0, 0.0)).to(DEV)   # 6 chunks, no polar pair
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, ninv, 1e-3)
    gen = torch.Generator(device=DEV).manual_seed(3)
    x = torch.view_as_complex(torch.randn(R, 2, p.ntri, 2, device=DEV, generator=gen))
    x[:, :, :L + 1] = x[:, :, :L + 1].real.to(x.dtype)
    u = torch.randn(R, 2, 12 * N * N, device=DEV, generator=gen)
    y = A.akra_apply_H(p, A.F32, x)
    b = A.akra_apply_At(p, A.F32, u, weighted=True)
    phi = R * (4 * N - 1) * (2 * L + 1) * 8
    tables = A.akra_plan_describe(A.akra_plan_create(N, L))["device_bytes"]
    # 33 right-hand sides at once are 6 chunks x 33 x 34 MB = 6.7 GB
    assert A.akra_plan_describe(p)["device_bytes"] - tables - phi <= 4 << 30
    for r in (0, 16, 17, 32):   # the edges of two groups
        assert torch.equal(A.akra_apply_H(p, A.F32, x[r:r + 1].contiguous())[0], y[r]), ("H", r)
        assert torch.equal(A.akra_apply_At(p, A.F32, u[r:r + 1].contiguous(), weighted=True)[0], b[r]), ("At", r)
