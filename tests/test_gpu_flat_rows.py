"""Row FFTs of the flat-sky operators at every decomposition of n: 16-point passes alone (n = 16^a), with a last
pass of 2, 4 or 8, from one pass to four; rows per block from 32 down to 1, joined into transposed stores or, at
n = 8192, transposed by a kernel of their own.

Tolerances are those of the operator tests: FP64 rel. L2 1e-10, FP32 2e-6 log2(n)."""
import math

import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("prec", [A.F64, A.F32])
@pytest.mark.parametrize("n", [16, 32, 128, 512, 1024, 4096, 8192])
def test_row_decompositions(n, prec):
    rng = np.random.default_rng(n)
    R = 1 if n > 1024 else 3
    p = A.akra_flat_plan_create(n)
    ninv = rng.uniform(0.5, 2.0, size=n * n) * (rng.uniform(size=n * n) < 0.7)
    A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
    w = O.FlatWeights(ninv.reshape(n, n), 1e-3)
    cdt, rdt = (torch.complex128, torch.float64) if prec == A.F64 else (torch.complex64, torch.float32)
    tol = 1e-10 if prec == A.F64 else 2e-6 * math.log2(n)
    x = rng.normal(size=(R, n, n)) + 1j * rng.normal(size=(R, n, n))
    xd = torch.from_numpy(x).to(DEV, cdt)
    h = A.akra_apply_H(p, prec, xd).to(torch.complex128).cpu().numpy()
    g = A.akra_apply_A(p, prec, xd).double().cpu().numpy()
    u = rng.normal(size=(R, 2, n * n))
    a = A.akra_apply_At(p, prec, torch.from_numpy(u).to(DEV, rdt)).to(torch.complex128).cpu().numpy()
    for r in range(R):
        assert rel(h[r], O.flat_apply_H(n, w, x[r])) < tol, ("H", r)
        g1, g2 = O.flat_forward_A(n, x[r])
        assert rel(g[r], np.stack([g1.ravel(), g2.ravel()])) < tol, ("A", r)
        assert rel(a[r], O.flat_adjoint_A(n, u[r][0].reshape(n, n), u[r][1].reshape(n, n))) < tol, ("At", r)
