"""The workspace memory that the library keeps between calls: at most a sixteenth of the device, given
back on request (and taken again by the next call with the same results), and given back by itself
when a call needs it in another shape while the rest of the device is full."""
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import RUN_SEED, sample_ids

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MB = 1 << 20


def _level(level, N, batch=0):
    cfg = mg.make_mlmc_cfg(RUN_SEED, 1.0, 0.3, 32, n0=17, rtol=1e-2, max_batch=batch)
    return mg.mlmc_level_estimate(cfg, level, int(sample_ids(level, 0, 1)[0]), N)[1]


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_kept_memory_is_bounded_and_given_back():
    mg.release_memory()
    Y = _level(2, 64, 64)  # some 2 GB of workspace
    mg.release_memory()
    before = _free()
    assert (Y == _level(2, 64, 64)).all()
    kept = before - _free()
    total = torch.cuda.mem_get_info()[1]
    assert 512 * MB < kept <= total // 16 + 64 * MB
    mg.release_memory()
    assert abs(_free() - before) <= 64 * MB
    assert (Y == _level(2, 64, 64)).all()
    mg.release_memory()


def test_kept_memory_serves_another_shape_on_a_full_device():
    mg.release_memory()
    ref = _level(3, 16, 16)
    mg.release_memory()
    _level(2, 256, 256)  # several GB in pieces of one size
    kept = _free()
    filler = torch.empty(kept - 1024 * MB, dtype=torch.uint8, device="cuda")
    try:
        assert (ref == _level(3, 16, 16)).all()  # needs more than the gigabyte that is left
        assert (ref == _level(3, 16)).all()      # the batch chosen from the memory there is
    finally:
        del filler
        mg.release_memory()
        torch.cuda.empty_cache()


def test_release_while_another_thread_solves():
    import threading

    n, B = 33, 8
    gen = torch.Generator(device="cuda").manual_seed(2)
    k = torch.exp(0.5 * torch.randn((B, n, n, n), generator=gen, dtype=torch.float64, device="cuda"))
    out, errors = [], []
    torch.cuda.synchronize()

    def work():
        st = torch.cuda.Stream()  # a created stream: every solve captures its cycle
        try:
            for _ in range(30):
                u = torch.zeros_like(k)
                torch.cuda.current_stream().synchronize()
                mg.mg_solve_batch(mg.mg_cfg(2, 2, 1e-8, 50, mg.MLMC_PREC_F64, engine=mg.MLMC_ENGINE_BATCHED), k, u,
                                  stream=st)
                out.append(u)
        except Exception as e:  # noqa: BLE001 (reported by the assertion below)
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    calls = 0
    while t.is_alive():
        mg.release_memory()
        calls += 1
    t.join()
    assert not errors and calls > 0
    assert all(torch.equal(u, out[0]) for u in out) and len(out) == 30
