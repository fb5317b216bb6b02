"""Workspace poisoning (test_gpu_poison.py) at band limits from 128 on over footprints of one hemisphere, where the
FP32 Legendre stages are the block-jump kernels: several chunks, several right-hand sides, the direct adjoint that
follows a block-jump synthesis, and rings up to a pole, whose pairs are in chunks of their own."""
import numpy as np
import pytest
import torch

import test_gpu_poison as P
from oracle import oracle as O
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("N,L,R,lo,hi", [(64, 130, 1, -0.95, -0.1), (64, 128, 3, -1.0, 0.05), (180, 150, 1, -0.95, -0.02)])
def test_results_do_not_depend_on_workspace_contents(N, L, R, lo, hi):
    rng = np.random.default_rng(N + L)
    z = np.cos(O.pixel_angles(N)[0])
    ninv = np.where((z > lo) & (z < hi), rng.uniform(200, 400, 12 * N * N), 0.0)
    p = A.akra_plan_create(N, L)
    A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
    x = torch.view_as_complex(torch.from_numpy(rng.normal(size=(R, 2, p.ntri, 2))).to(DEV))
    x[:, :, :L + 1] = x[:, :, :L + 1].real.to(x.dtype)
    y = A.akra_apply_A(p, A.F64, x) * torch.from_numpy(ninv > 0).to(DEV)
    first = P._calls(p, x, y)
    A.akra_plan_fill_workspaces(p, 0xFF)
    torch.cuda.synchronize()
    second = P._calls(p, x, y)
    for k in first:
        a, b = first[k], second[k]
        assert bool(torch.isfinite(torch.view_as_real(b) if b.is_complex() else b).all()), k
        assert torch.equal(a, b), k
