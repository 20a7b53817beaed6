"""The small-grid engine's 17^3 form (one sample per SM) at the sizes where its work queue and its
choice change: one sample, one per SM, one more than that, against the batched kernels bit for bit."""
import numpy as np
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import random_coefficient, random_rhs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("extra", [None, 0, 1])
@pytest.mark.parametrize("prec,accel", [(mg.MLMC_PREC_F64, mg.MLMC_ACCEL_NONE), (mg.MLMC_PREC_F64, mg.MLMC_ACCEL_CG),
                                        (mg.MLMC_PREC_MIXED, mg.MLMC_ACCEL_NONE),
                                        (mg.MLMC_PREC_MIXED, mg.MLMC_ACCEL_CG)])
@pytest.mark.parametrize("nu", [(2, 2), (1, 3)])
def test_engine17_equals_batched_bitwise(prec, accel, nu, extra):
    B = 1 if extra is None else torch.cuda.get_device_properties(0).multi_processor_count + extra
    k = torch.from_numpy(np.stack([random_coefficient(17, 300 + s, 0.2 + 0.3 * (s % 4)) for s in range(B)])).cuda()
    f = torch.from_numpy(np.stack([random_rhs(17, 700 + s) for s in range(B)])).cuda()
    out = []
    for engine in (mg.MLMC_ENGINE_BATCHED, mg.MLMC_ENGINE_CTA):
        u = torch.zeros_like(k)
        cyc, rel, st = mg.mg_solve_batch(
            mg.mg_cfg(nu[0], nu[1], 1e-9, 100, prec, mg.MLMC_SMOOTH_TWO_PASS, accel, engine=engine), k, u, f,
            allow_not_converged=True)  # the plain cycle diverges on the roughest of these
        out.append((u.cpu().numpy(), cyc, rel, st))
    assert np.array_equal(out[0][1], out[1][1]) and out[0][3] == out[1][3]
    assert np.array_equal(out[0][2], out[1][2], equal_nan=True)
    assert np.array_equal(out[0][0], out[1][0], equal_nan=True)
