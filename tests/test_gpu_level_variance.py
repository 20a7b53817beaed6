"""Level statistics of samples that do not differ, or hardly do: the variance is zero for identical
samples (a field of variance zero makes them so) and never negative, wherever a batch ends, and M2
is that of the samples in 64-bit two-pass arithmetic for ordinary ones."""
import math

import numpy as np
import pytest

import paper_1607_03252_gb300 as mg
from paper_1607_03252_gb300.workloads import RUN_SEED, sample_ids

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rtol", [1e-4, 1e-7, 1e-8, 1e-9, 1e-10])
@pytest.mark.parametrize("level", [0, 1])
@pytest.mark.parametrize("N,batch", [(1, 0), (2, 0), (33, 0), (333, 0), (333, 50), (1500, 700)])
def test_identical_samples_have_no_variance(level, rtol, N, batch):
    cfg = mg.make_mlmc_cfg(RUN_SEED, 0.0, 0.3, 8, n0=9, rtol=rtol, max_batch=batch)
    st, Y, *_ = mg.mlmc_level_estimate(cfg, level, 5, N)
    assert len(set(Y.tolist())) == 1
    assert st.M2 == 0.0 and st.var_biased == 0.0 and st.var_unbiased == 0.0
    assert abs(st.mean - Y[0]) <= 2.0 ** -52 * abs(Y[0])


@pytest.mark.parametrize("sigma2", [1e-32, 1e-31, 1e-30, 1e-20, 1.0])
def test_variance_is_that_of_the_samples(sigma2):
    N = 300
    cfg = mg.make_mlmc_cfg(RUN_SEED, sigma2, 0.3, 64, n0=9, rtol=1e-10, max_batch=77)
    st, Y, *_ = mg.mlmc_level_estimate(cfg, 0, int(sample_ids(0, 3, 1)[0]), N)
    exact = [float(y) for y in Y]
    mean = math.fsum(exact) / N
    M2 = math.fsum((y - mean) ** 2 for y in exact)
    # each product carries a few roundings of t, and t those of a product and two sums: relative
    # 1e-14 of M2, and N deviations of an ulp of the mean
    assert st.M2 >= 0.0
    assert abs(st.M2 - M2) <= 1e-14 * N * M2 + N * (2.0 ** -51 * abs(mean)) ** 2 + 2.0 ** -50 * abs(mean) * math.sqrt(N * M2)
    assert np.isfinite(st.var_unbiased)
