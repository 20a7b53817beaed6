"""The convergence test that goes along with the next cycle's first red pass: samples that turn out
to be done get their replaced values back, samples that go on after all take the pass on its own.
With a tolerance at the reported residual of cycle c the sample stops after it, with one just below
it goes on; the iterates are compared bit for bit with those of fixed cycles, which take no test in
between, from early cycles down to the rounding level."""
import numpy as np
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import random_coefficient, random_rhs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve(k, f, rtol, maxc, sm, engine):
    u = torch.zeros_like(k)
    cyc, rel, _ = mg.mg_solve_batch(mg.mg_cfg(2, 2, rtol, maxc, mg.MLMC_PREC_F64, sm, engine=engine), k, u, f,
                                    allow_not_converged=True)
    return u.cpu().numpy(), cyc, rel


@pytest.mark.parametrize("n,sm,engine", [(17, mg.MLMC_SMOOTH_SPLIT, mg.MLMC_ENGINE_BATCHED),
                                         (33, mg.MLMC_SMOOTH_SPLIT, mg.MLMC_ENGINE_BATCHED),
                                         (65, mg.MLMC_SMOOTH_SPLIT, mg.MLMC_ENGINE_BATCHED),
                                         (33, mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_ENGINE_BATCHED),
                                         (17, mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_ENGINE_CTA),
                                         (33, mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_ENGINE_CTA)])
def test_tolerance_at_the_residual_of_a_cycle(n, sm, engine):
    B = 3
    k = torch.from_numpy(np.stack([random_coefficient(n, 40 + s, 0.5 + 0.4 * s) for s in range(B)])).cuda()
    f = torch.from_numpy(np.stack([random_rhs(n, 60 + s) for s in range(B)])).cuda()
    fixed = {c: _solve(k, f, 0.0, c, sm, engine) for c in (3, 4, 14, 15, 22, 23)}
    for c in (3, 14, 22):
        for s in range(B):
            r = float(fixed[c][2][s])
            if not r < 1.0:  # the cycle does not converge on this sample: no tolerance to set
                continue
            # at its own residual a sample stops after cycle c (or earlier, where it stagnates)
            u, cyc, rel = _solve(k[s:s + 1], f[s:s + 1], r * (1.0 + 1e-13), 40, sm, engine)
            assert cyc[0] <= c and rel[0] <= r * (1.0 + 1e-13)
            if cyc[0] == c:
                assert np.array_equal(u[0], fixed[c][0][s]) and rel[0] == r
            # just below it the sample goes on for one cycle more
            for below in (1e-15, 1e-9, 1e-4):
                u, cyc, rel = _solve(k[s:s + 1], f[s:s + 1], r * (1.0 - below), c + 1, sm, engine)
                if cyc[0] == c + 1:
                    assert np.array_equal(u[0], fixed[c + 1][0][s]) and rel[0] == fixed[c + 1][2][s]
                else:
                    assert cyc[0] < c and rel[0] <= r
