"""Run by tests/test_gpu_debug_block_jump.py in a child process whose AKRA_LIBRARY names the bounds-checked
build: the operators at band limits from 128 on over footprints of one hemisphere, where the FP32 Legendre
stages advance by blocks of 16 steps (csrc/akra_legendre_blk.cuh), against the FP64 oracle, then the
library's record of out-of-bounds indices and of barriers left open.  Prints one JSON line."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402
import torch  # noqa: E402

from oracle import oracle as O  # noqa: E402
import synthetic as S  # noqa: E402
from paper_2606_06175_gb300 import akra as A  # noqa: E402


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


def main():
    dev = torch.device("cuda:0")
    out = {"library": os.path.basename(A.library_path()), "errors": {}}
    A.akra_debug_violations()   # start from a clear record
    # one tile and a bit, several tiles with a ragged end, more than one chunk of rings, rings up to a pole
    for N, L, R, sky in ((64, 128, 2, "south"), (64, 131, 1, "north_pole"), (100, 301, 2, "south"), (180, 160, 1, "south")):
        rng = np.random.default_rng(N + L)
        z = np.cos(O.pixel_angles(N)[0])
        fp = (z < -0.1) & (z > -0.95) if sky == "south" else z > 0.2
        ninv = np.where(fp, 1.0 + rng.random(12 * N * N), 0.0)
        w = O.Weights(N, ninv, 1e-3)
        tol = 4 * 2.0 ** -24 * L
        p = A.akra_plan_create(N, L)
        A.akra_plan_set_weights(p, torch.from_numpy(ninv).to(dev), 1e-3)
        pairs = [(S.random_alm(L, rng), S.random_alm(L, rng)) for _ in range(R)]
        x = torch.from_numpy(np.stack([np.stack(q) for q in pairs])).to(dev, torch.complex64)
        u = rng.normal(size=(R, 2, 12 * N * N)).astype(np.float32)
        h = [np.stack(O.apply_H(N, L, w, *q)) for q in pairs]
        bt = A.akra_batch_create([p], [R])
        got = {"H": A.akra_apply_H(p, A.F32, x), "batch": A.akra_batch_apply_H(bt, [x])[0],
               "At": A.akra_apply_At(p, A.F32, torch.from_numpy(u).to(dev), weighted=True)}
        for name, y in got.items():
            for r in range(R):
                ref = h[r] if name != "At" else np.stack(O.rhs_b(N, L, w, *u[r].astype(np.float64)))
                e = rel(y[r].to(torch.complex128).cpu().numpy(), ref)
                out["errors"]["%s_%d_%d_%d" % (name, N, L, r)] = e
                assert e < tol, (name, N, L, r, e)
        del bt
    torch.cuda.synchronize()
    out["violations"] = A.akra_debug_violations()
    print(json.dumps(out))


if __name__ == "__main__":
    main()
