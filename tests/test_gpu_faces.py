"""The set-up's FP64 quotients: a solve with the coefficient scaled by a power of two scales the
solution by its inverse exactly, whichever division the set-up takes. Scaled by 2^200 or 2^-200
the faces and 1/D come from the language's division, unscaled from the short one: the iterates
agree bit for bit only if every quotient does."""
import numpy as np
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import random_coefficient

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sm", [mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_SMOOTH_SPLIT])
@pytest.mark.parametrize("n", [9, 33, 65])
def test_scaled_coefficient_scales_the_solution_exactly(n, sm):
    k = torch.from_numpy(np.stack([random_coefficient(n, 70 + s, 1.0) for s in range(2)])).cuda()
    out = []
    for e in (0, 200, -200):
        u = torch.zeros_like(k)
        cfg = mg.mg_cfg(2, 2, 0.0, 2, mg.MLMC_PREC_F64, sm, engine=mg.MLMC_ENGINE_BATCHED)
        mg.mg_solve_batch(cfg, k * 2.0 ** e, u)
        out.append((u * 2.0 ** e).cpu().numpy())
    assert np.isfinite(out[0]).all() and np.abs(out[0]).max() > 0
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
