"""Second moments of observations near the origin under states whose means are far
from it (a start that does not fit yet, an outlier): the sums are of x^2, xy and
y^2 as the header says, and keep their own digits. They are compared with the 64-bit
sums over the very rows that hmm_posterior returns; products and sums keep what
FP32 drops, 2^-46 a term: bar 1e-9 of every entry.
"""
import numpy as np
import pytest
import torch

from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [2, 8, 65, 5000])
@pytest.mark.parametrize("K", [1, 3, 9, 32])
def test_moments_near_the_origin(cuda_lib, K, T):
    api = cuda_lib
    rng = np.random.default_rng(10 * K + T)
    prm = synth.random_params(K, rng)
    prm.mu[:] = (250.0, 140.0) + rng.normal(0, 1, (K, 2)).astype(np.float32)
    prm.cov[:] = (2500.0, 0.0, 1600.0)
    fl = (rng.random(T) < 0.3).astype(np.uint8)
    fl[0] = 1
    xy = (rng.uniform(0.1, 0.9, (T, 2)) * fl[:, None]).astype(np.float32)
    dev, dxy, dfl = api.to_device(prm), torch.from_numpy(xy).cuda(), torch.from_numpy(fl).cuda()
    ctx = api.Context()
    try:
        st, _ = ctx.hmm_expected_stats(*dev, dxy, dfl)
        g, _ = ctx.hmm_posterior(*dev, dxy, dfl)
        st = {k: v.cpu().numpy() for k, v in st.items()}
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    g = g.cpu().numpy().astype(np.float64) * fl[:, None]
    x, y = xy.astype(np.float64).T
    for name, w in (("Gr", fl), ("Sx", x), ("Sy", y), ("Sxx", x * x), ("Sxy", x * y), ("Syy", y * y)):
        np.testing.assert_allclose(st[name], w @ g, rtol=1e-9, atol=0, err_msg=name)
