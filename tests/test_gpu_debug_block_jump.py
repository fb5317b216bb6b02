"""The bounds-checked build over the block-jump Legendre kernels (lmax >= 128 on footprints of one hemisphere,
which test_gpu_debug_build.py's small plans do not reach): no out-of-bounds index, and no barrier of a block
whose last phase is still open when the block ends -- an arrival of the tensor core after that would land in
the shared memory of the next block."""
import json
import os
import subprocess
import sys

import pytest

from paper_2606_06175_gb300 import build as B

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_block_jump_kernels_record_no_violation():
    B.build()
    env = dict(os.environ, AKRA_LIBRARY=B.OUT_DEBUG)
    r = subprocess.run([sys.executable, os.path.join(HERE, "debug_block_jump_run.py")], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["library"] == "libakra_debug.so"
    assert out["violations"]["count"] == 0, out["violations"]
