"""Expired waits of the tcgen05 field kernel on every block shape (16, 32 and 64 x-values per block:
17^3, 33^3, 65^3) with one group sum and with folds (more than 256 features): the blocks of the
volume and of the face x = n - 1 give up, write NaN to their nodes and leave, the call reports
MLMC_ERR_TIMEOUT, and the same context then gives the field bit for bit. With a budget of 0 any
wait of any thread may be the one that gives up."""
import numpy as np
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import RUN_SEED, sample_ids

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(17, 5, 64), (17, 3, 300), (33, 3, 100), (33, 2, 300), (65, 2, 300), (65, 1, 8)]


@pytest.fixture
def restore_controls():
    yield
    mg.set_wait_budget(2_000_000_000)
    mg.inject_wait_failure(0)


def _field(n, B, M):
    k = torch.zeros((B, n, n, n), dtype=torch.float64, device="cuda")
    return mg.field_cfg(RUN_SEED, 1.0, 0.3, M), sample_ids(2, 11, B), k


@pytest.mark.parametrize("n,B,M", SHAPES)
def test_injected_wait_failure(restore_controls, n, B, M):
    fc, ids, ref = _field(n, B, M)
    mg.mlmc_field_eval(fc, ids, ref)
    mg.set_wait_budget(100_000)
    mg.inject_wait_failure(1)
    k = torch.zeros_like(ref)
    with pytest.raises(mg.MlmcError) as e:
        mg.mlmc_field_eval(fc, ids, k)
    assert e.value.status == mg.MLMC_ERR_TIMEOUT
    edge = torch.zeros((n, n, n), dtype=torch.bool, device="cuda")
    edge[:, n - 1, n - 1] = True  # x = y = n - 1 is another kernel's
    assert torch.isnan(k[:, ~edge]).all() and torch.equal(k[:, edge], ref[:, edge])
    mg.set_wait_budget(2_000_000_000)
    again = torch.zeros_like(ref)
    mg.mlmc_field_eval(fc, ids, again)
    assert torch.equal(again, ref)


@pytest.mark.parametrize("n,B,M", SHAPES)
def test_no_time_to_wait(restore_controls, n, B, M):
    fc, ids, ref = _field(n, B, M)
    mg.mlmc_field_eval(fc, ids, ref)
    mg.set_wait_budget(0)
    for _ in range(5):
        k = torch.zeros_like(ref)
        with pytest.raises(mg.MlmcError) as e:
            mg.mlmc_field_eval(fc, ids, k)
        assert e.value.status == mg.MLMC_ERR_TIMEOUT
        ok = (k == ref) | torch.isnan(k)
        assert ok.all()  # a node is its value or NaN, nothing else
    mg.set_wait_budget(2_000_000_000)
    again = torch.zeros_like(ref)
    mg.mlmc_field_eval(fc, ids, again)
    assert torch.equal(again, ref)
