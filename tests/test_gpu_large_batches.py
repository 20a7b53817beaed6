"""Batches above half the launch limit of 65535 samples on the colour-split storage, with and without
post-smoothing: bit for bit the nodal sweep's iterates."""
import pytest

import paper_1607_03252_gb300 as mg

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [(2, 0), (1, 1)])
@pytest.mark.parametrize("B", [32767, 32768, 65535])
def test_split_storage_takes_every_batch(B, nu):
    n = 9
    gen = torch.Generator(device="cuda").manual_seed(B)
    k = torch.exp(0.3 * torch.randn((B, n, n, n), generator=gen, dtype=torch.float64, device="cuda"))
    out = []
    for sm in (mg.MLMC_SMOOTH_NODAL, mg.MLMC_SMOOTH_SPLIT):
        u = torch.zeros_like(k)
        cfg = mg.mg_cfg(nu[0], nu[1], 0.0, 2, mg.MLMC_PREC_MIXED, sm, engine=mg.MLMC_ENGINE_BATCHED)
        mg.mg_solve_batch(cfg, k, u)
        out.append(u)
    assert out[0].abs().max() > 0 and torch.equal(out[0], out[1])
