"""Cycle counts on rough coefficients (lognormal, variance 2 to 6): the convergence test that comes with
the next cycle's first red pass (colour-split storage, the small-grid engine at 33^3), the one on the
red residuals alone (plain storage) and the full one agree, with tolerances at and just above the
residual of a cycle from early ones down to the smallest tolerance that the merged test takes,
2^-51 (n - 1)^2; every solve is compared, and enough of them lie close to that tolerance."""
import math

import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import RUN_SEED, sample_ids

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FORMS = [(mg.MLMC_SMOOTH_SPLIT, mg.MLMC_ENGINE_BATCHED), (mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_ENGINE_BATCHED),
         (mg.MLMC_SMOOTH_TWO_PASS, mg.MLMC_ENGINE_CTA)]


def _solve(k, f, rtol, cycles, form):
    u = torch.zeros_like(k)
    cfg = mg.mg_cfg(2, 2, rtol, cycles, mg.MLMC_PREC_F64, form[0], engine=form[1])
    cyc, rel, _ = mg.mg_solve_batch(cfg, k, u, f, allow_not_converged=True)
    return u, cyc, rel


@pytest.mark.parametrize("sigma2", [2.0, 4.0, 6.0])
@pytest.mark.parametrize("n", [17, 33])
def test_every_form_stops_after_the_same_cycle(n, sigma2):
    B, floor = 4, 2.0 ** -51 * (n - 1) ** 2
    k = torch.empty((B, n, n, n), dtype=torch.float64, device="cuda")
    mg.mlmc_field_eval(mg.field_cfg(RUN_SEED, sigma2, 0.25, 128), sample_ids(3, 40, B), k)
    gen = torch.Generator(device="cuda").manual_seed(n)
    f = torch.rand(k.shape, generator=gen, dtype=torch.float64, device="cuda") * 2.0 - 1.0
    f[0] = 1.0
    # residuals after fixed cycles, by the full test
    after = {c: _solve(k, f, 0.0, c, FORMS[1])[2] for c in range(6, 50)}
    near = 0
    for s in range(B):
        for c, rel in after.items():
            r = float(rel[s])
            if not (math.isfinite(r) and floor <= r < 1e4 * floor):
                continue
            for factor in (1.0 + 1e-13, 1.1, 1.2):
                out = [_solve(k[s:s + 1], f[s:s + 1], r * factor, 60, form) for form in FORMS]
                assert len({int(o[1][0]) for o in out}) == 1
                assert len({float(o[2][0]) for o in out}) == 1 and out[0][2][0] <= r * factor
                assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][0], out[2][0])
                near += 1
    assert near >= 12
