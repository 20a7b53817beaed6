"""The 5^3 grid alone (one dense solve, no sweep) with the colour-split storage asked for: the
solution and the residual that is reported are the two-pass form's."""
import numpy as np
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import random_coefficient

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [mg.MLMC_PREC_F64, mg.MLMC_PREC_MIXED])
def test_split_storage_on_the_smallest_grid(prec):
    k = torch.from_numpy(np.stack([random_coefficient(5, 40 + s, 1.0) for s in range(3)])).cuda()
    out = []
    for sm in (mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_SMOOTH_SPLIT):
        u = torch.zeros_like(k)
        cyc, rel, st = mg.mg_solve_batch(mg.mg_cfg(2, 2, 1e-10, 20, prec, sm, engine=mg.MLMC_ENGINE_BATCHED), k, u)
        assert st == mg.MLMC_OK
        out.append((u.cpu().numpy(), cyc, rel))
    assert all(np.array_equal(a, b) for a, b in zip(*out))
