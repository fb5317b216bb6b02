"""A batch's captured iteration and its work lists: a solve after the lists have been rebuilt (another synthesis
group and back, another tile shape by the tuner) uses the new ones.  The captured iteration of the first
solve holds the addresses of lists that are released in between."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
import synthetic as S
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _batch(rng):
    plans, shears = [], []
    for N, L, R in ((16, 40, 5), (64, 128, 4)):     # from the queues; block jumps unless the group takes them
        z = np.cos(O.pixel_angles(N)[0])
        ninv = np.where((z < 0.05) & (z > -0.9), rng.uniform(200, 400, 12 * N * N), 0.0)
        p = A.akra_plan_create(N, L)
        A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
        y = np.stack([np.stack(O.forward_A(N, L, S.random_alm(L, rng), S.random_alm(L, rng))) for _ in range(R)])
        y = np.where(ninv > 0, y + 0.05 * rng.normal(size=y.shape), 0.0)
        plans.append(p)
        shears.append(torch.from_numpy(y).to(DEV))
    return A.akra_batch_create(plans, [5, 4]), plans, shears


def test_solve_after_the_work_lists_were_rebuilt():
    rng = np.random.default_rng(5)
    b, plans, shears = _batch(rng)
    single = [A.akra_cg_solve(p, A.MIXED, y, tol=1e-10, maxiter=3000)[0] for p, y in zip(plans, shears)]

    def check(what):
        xs, infos = A.akra_batch_cg_solve(b, A.MIXED, shears, tol=1e-10, maxiter=3000)
        for x, ref, info in zip(xs, single, infos):
            assert info["status"] == 0, (what, info)
            # two solutions at relative residual 1e-10, condition number at most (400 + λ) / λ with λ = 1e-3 · 300
            assert float((x - ref).norm() / ref.norm()) < 2 * 1e-10 * 1334, what

    A.akra_batch_set_tc_synthesis(b, 4)
    check("first")
    A.akra_batch_set_tc_synthesis(b, 8)
    A.akra_batch_set_tc_synthesis(b, 4)
    check("same group, new list")
    A.akra_batch_autotune(b)
    check("tuned")
    A.akra_batch_autotune(b)
    check("tuned again")
