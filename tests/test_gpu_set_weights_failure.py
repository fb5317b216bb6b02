"""akra_plan_set_weights that fails: the plan then has no weights, instead of some of the new ones under the
old λ_eff and ring lists, until a later call succeeds; and a call that succeeds allocates no table, so that it
cannot run out of memory half-way (an FP32 H without the tables of its ring list was λ x with status OK)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _sphere():
    N, L = 64, 128
    z = np.cos(O.pixel_angles(N)[0])
    return A.akra_plan_create(N, L), torch.from_numpy(np.where((z < -0.1) & (z > -0.9), 2.0, 0.0)).to(DEV)


def _flat():
    n = 32
    return A.akra_flat_plan_create(n), torch.full((n * n,), 2.0, dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("make", [_sphere, _flat])
def test_failed_set_weights_leaves_no_weights(make):
    p, ninv = make()
    A.akra_plan_set_weights(p, ninv, 1e-3)
    x = torch.ones(p.alm_shape(1), dtype=torch.complex64, device=DEV)
    y = A.akra_apply_H(p, A.F32, x)
    b = A.akra_batch_create([p], [1]) if make is _sphere else None
    bad = 2 * ninv
    bad[-1] = -1.0
    with pytest.raises(A.AkraError) as ei:
        A.akra_plan_set_weights(p, bad, 1e-3)
    assert ei.value.status == 1   # EINVAL
    calls = [lambda: A.akra_apply_H(p, A.F32, x)]
    if b is not None:
        calls.append(lambda: A.akra_batch_apply_H(b, [x]))
    for call in calls:
        with pytest.raises(A.AkraError) as ei:
            call()
        assert ei.value.status == 7   # ENOWEIGHTS
    A.akra_plan_set_weights(p, ninv, 1e-3)
    assert torch.equal(A.akra_apply_H(p, A.F32, x), y)


def test_set_weights_allocates_no_table():
    p, ninv = _sphere()
    before = A.akra_plan_describe(p)["device_bytes"]
    A.akra_plan_set_weights(p, ninv, 1e-3)
    assert A.akra_plan_describe(p)["device_bytes"] == before
