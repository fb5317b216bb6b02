"""Device memory of a solve whose tensor-core synthesis group is set: the group's staged operand is held only where
the tensor-core kernel runs (not on a footprint of one hemisphere with groups of 4 and 8)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("group,held", [(4, False), (8, False), (16, True)])
def test_solve_holds_the_operand_only_where_it_is_used(group, held):
    N, L, R = 64, 128, 4
    z = np.cos(O.pixel_angles(N)[0])
    ninv = torch.from_numpy(np.where((z < -0.1) & (z > -0.9), 200.0, 0.0)).to(DEV)
    y = torch.randn(R, 2, 12 * N * N, device=DEV, generator=torch.Generator(device=DEV).manual_seed(2)) * (ninv > 0)
    held_bytes = []
    for g in (0, group):
        p = A.akra_plan_create(N, L)
        A.akra_plan_set_weights(p, ninv, 1e-3)
        A.akra_plan_set_tc_synthesis(p, R, g)
        _, info = A.akra_cg_solve(p, A.F32, y.float(), tol=1e-4, maxiter=2000)
        assert info["status"] == 0, info
        held_bytes.append(A.akra_plan_describe(p)["device_bytes"])
    assert (held_bytes[1] > held_bytes[0]) == held
