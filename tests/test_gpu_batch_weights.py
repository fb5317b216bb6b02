"""A batch whose plans get new weights: its work lists follow the footprint.  Footprints grow and shrink in
ring pairs past a chunk of 128, on a plan whose Legendre stages run from the batch's queues and on one whose
stages are block-jump launches of their own, with the CUDA-core and the tensor-core synthesis."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
import synthetic as S
from paper_2606_06175_gb300 import akra as A

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
SPEC = [(100, 60, 2), (64, 128, 3)]                     # (Nside, lmax, R): queue, block jumps
BANDS = [(-0.55, -0.45), (-0.93, 0.02), (-0.7, -0.6), (-0.4, 0.4)]   # the last needs both rings of every pair


def tol32(lmax):
    return 4 * 2.0 ** -24 * max(lmax, 16)   # as in test_gpu_batch.py


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _ninv(N, band, rng):
    z = np.cos(O.pixel_angles(N)[0])
    return np.where((z > band[0]) & (z < band[1]), 1.0 + rng.random(12 * N * N), 0.0)


@pytest.mark.parametrize("group", [0, 4])
def test_batched_H_follows_new_weights(group):
    rng = np.random.default_rng(17 + group)
    plans = [A.akra_plan_create(N, L) for N, L, _ in SPEC]
    pairs = [[(S.random_alm(L, rng), S.random_alm(L, rng)) for _ in range(R)] for _, L, R in SPEC]
    xs = [torch.from_numpy(np.stack([np.stack(q) for q in pr])).to(DEV, torch.complex64) for pr in pairs]
    b = None
    for band in BANDS:
        w = []
        for (N, L, R), p in zip(SPEC, plans):
            ninv = _ninv(N, band, rng)
            A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(DEV), 1e-3)
            w.append(O.Weights(N, ninv, 1e-3))
        if b is None:
            b = A.akra_batch_create(plans, [R for *_, R in SPEC])
            A.akra_batch_set_tc_synthesis(b, group)
        ys = A.akra_batch_apply_H(b, xs)
        for i, (N, L, R) in enumerate(SPEC):
            for r in range(R):
                ref = np.stack(O.apply_H(N, L, w[i], *pairs[i][r]))
                assert rel(ys[i][r].cpu().numpy(), ref) < tol32(L), (band, N, r)
