"""The small-grid engine's 17^3 form with several samples to every SM's block (each block takes one
after the other from the queue and reuses its shared memory), mixed refinement and mixed CG, and FP64
up to one sample per SM: bit for bit the batched kernels, and the same when it is run again."""
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import RUN_SEED, sample_ids

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _solve(k, prec, accel, engine):
    u = torch.zeros_like(k)
    cfg = mg.mg_cfg(2, 2, 1e-10, 100, prec, mg.MLMC_SMOOTH_TWO_PASS, accel, engine=engine)
    cyc, rel, st = mg.mg_solve_batch(cfg, k, u, allow_not_converged=True)
    return u, cyc, rel, st


@pytest.mark.parametrize("prec,accel,per_sm", [(mg.MLMC_PREC_MIXED, mg.MLMC_ACCEL_NONE, 5),
                                               (mg.MLMC_PREC_MIXED, mg.MLMC_ACCEL_CG, 5),
                                               (mg.MLMC_PREC_F64, mg.MLMC_ACCEL_NONE, 1),
                                               (mg.MLMC_PREC_F64, mg.MLMC_ACCEL_CG, 1)])
def test_queue_equals_batched_bitwise_every_time(prec, accel, per_sm):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = per_sm * sms + (37 if per_sm > 1 else 0)
    k = torch.empty((B, 17, 17, 17), dtype=torch.float64, device="cuda")
    mg.mlmc_field_eval(mg.field_cfg(RUN_SEED, 1.5, 0.2, 64), sample_ids(0, 100, B), k)
    ub, cb, rb, sb = _solve(k, prec, accel, mg.MLMC_ENGINE_BATCHED)
    for _ in range(3):
        u, c, r, st = _solve(k, prec, accel, mg.MLMC_ENGINE_CTA)
        assert st == sb and (c == cb).all() and (r == rb).all()
        assert torch.equal(u, ub)
