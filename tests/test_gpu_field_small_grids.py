"""The tcgen05 field on the grids below 65^3 (16 and 32 x-values per block) against the warp-level
mma.sync form, bit for bit: both form the same slices and exact group sums. Several samples, feature
counts that are no multiple of a k-step's eight, more than one fold, and FP32 output. The arithmetic
is chosen by MLMC_FIELD_ARITH, read once per process, so each form runs in a child process."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

DUMP = r"""
import sys, numpy as np, torch
import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import RUN_SEED, sample_ids
out = {}
for n, B, M, cov in ((17, 1, 8, 0), (17, 7, 100, 1), (17, 2, 257, 0), (17, 3, 1000, 0), (33, 1, 3, 0), (33, 5, 100, 1),
                     (33, 2, 513, 0)):
    for name, dtype in (("f64", torch.float64), ("f32", torch.float32)):
        k = torch.empty((B, n, n, n), dtype=dtype, device="cuda")
        mg.mlmc_field_eval(mg.field_cfg(RUN_SEED, 1.0, 0.2, M, cov), sample_ids(3, 2, B), k)
        out["%d_%d_%d_%s" % (n, B, M, name)] = k.cpu().numpy()
np.savez(sys.argv[1], **out)
"""


def test_small_grids_match_warp_mma_bitwise(tmp_path):
    res = {}
    for arith in (3, 4):
        f = tmp_path / ("k%d.npz" % arith)
        env = dict(os.environ, MLMC_FIELD_ARITH=str(arith))
        r = subprocess.run([sys.executable, "-c", DUMP, str(f)], cwd=ROOT, env=env, capture_output=True, text=True,
                           timeout=600)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
        res[arith] = dict(np.load(f))
    assert len(res[3]) == 14
    for key in res[3]:
        assert np.array_equal(res[3][key], res[4][key]), key
