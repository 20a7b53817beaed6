"""The V-cycle's red-black shortcuts (first red pass from a zero guess, residual and
restriction on the red nodes, interpolation to the black nodes) with and without pre- and
post-smoothing, on every storage and engine, against the FP64 oracle's full V-cycle."""
import numpy as np
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import random_coefficient, random_rhs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = [(mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_ENGINE_BATCHED), (mg.MLMC_SMOOTH_SPLIT, mg.MLMC_ENGINE_BATCHED),
         (mg.MLMC_SMOOTH_FUSED_32x8, mg.MLMC_ENGINE_BATCHED), (mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_ENGINE_CTA)]


def _inputs(n, B):
    k = np.stack([random_coefficient(n, 900 + s, 1.0) for s in range(B)])
    f = np.stack([random_rhs(n, 950 + s) for s in range(B)])
    return k, f


def _solve(k, f, cfg):
    u = torch.zeros(k.shape, dtype=torch.float64, device="cuda")
    cyc, rel, st = mg.mg_solve_batch(cfg, torch.from_numpy(k).cuda(), u, torch.from_numpy(f).cuda(),
                                     allow_not_converged=True)
    return u.cpu().numpy(), cyc, rel, st


@pytest.mark.parametrize("sm,engine", FORMS)
@pytest.mark.parametrize("nu", [(2, 2), (1, 0), (0, 2), (3, 1)])
@pytest.mark.parametrize("n", [5, 9, 17, 33])
def test_f64_cycles_match_oracle(orc, n, nu, sm, engine):
    k, f = _inputs(n, 2)
    u, cyc, rel, _ = _solve(k, f, mg.mg_cfg(nu[0], nu[1], 0.0, 3, mg.MLMC_PREC_F64, sm, engine=engine))
    for s in range(2):
        uo, _, _, ro, _ = orc.mg_solve(k[s], f[s], nu1=nu[0], nu2=nu[1], rtol=0.0, max_cycles=3)
        assert np.abs(u[s] - uo).max() <= 1e-10 * np.abs(uo).max()
        assert abs(rel[s] - ro) <= 1e-8 * max(ro, 1e-4)


@pytest.mark.parametrize("sm,engine", FORMS + [(mg.MLMC_SMOOTH_NODAL, mg.MLMC_ENGINE_BATCHED),
                                               (mg.MLMC_SMOOTH_NODAL, mg.MLMC_ENGINE_CTA)])
@pytest.mark.parametrize("accel,nu", [(mg.MLMC_ACCEL_NONE, (2, 2)), (mg.MLMC_ACCEL_CG, (0, 2)), (mg.MLMC_ACCEL_CG, (2, 0))])
@pytest.mark.parametrize("n", [9, 33])
def test_mixed_reaches_the_oracle_solution(orc, n, accel, nu, sm, engine):
    k, f = _inputs(n, 2)
    u, _, rel, st = _solve(k, f, mg.mg_cfg(nu[0], nu[1], 1e-12, 300, mg.MLMC_PREC_MIXED, sm, accel, engine=engine))
    assert st == mg.MLMC_OK and rel.max() <= 1e-12
    for s in range(2):
        uo, *_ = orc.mg_solve(k[s], f[s], rtol=1e-12, max_cycles=300)
        assert np.abs(u[s] - uo).max() <= 1e-9 * np.abs(uo).max()
