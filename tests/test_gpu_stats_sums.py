"""The E-step's sums lose nothing to the number of steps they are taken over.

Visits: Gs and Gr against the 64-bit sums of the very rows that hmm_posterior
returns. What the FP32 additions drop is kept beside them, so they agree to
2^-48 a term, 1e-10 of the sum; bar 1e-9 (FP32 sums over a block of steps: 1e-8).

Transitions: the rows of N add up to the visits but the last step's, in exact
arithmetic and in the oracle. The rounding of the model's constants moves both
alike (up to 1e-7 of them), so it drops out of the difference; left are the
roundings of a step's P u and of its scale, one or two of 2^-24, which a quiet
stretch repeats: bar 6e-8 of the largest entry.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [4, 8, 16, 25, 32, 50])
def test_sums(cuda_lib, K):
    api = cuda_lib
    rng = np.random.default_rng(K)
    gen = synth.random_params(K, rng)
    o = synth.sample_observations(gen, 100_003, rng)
    prm = synth.perturb_params(gen, rng)
    dev, xy, fl = api.to_device(prm), torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    ctx = api.Context()
    try:
        st, _ = ctx.hmm_expected_stats(*dev, xy, fl)
        assert ctx.last_chunk_proposals() == 0
        st = {k: v.cpu().numpy() for k, v in st.items()}
        g, _ = ctx.hmm_posterior(*dev, xy, fl)
        g = g.cpu().numpy().astype(np.float64)
    finally:
        ctx.close()
    for name, want in (("Gs", g.sum(0)), ("Gr", g[o.tremor > 0].sum(0))):
        assert np.abs(st[name] - want).max() <= 1e-9 * want.max(), name
    want, _ = oracle.expected_stats(prm, o.xy, o.tremor)
    off = (st["N"].sum(1) - want["N"].sum(1)) - (st["Gs"] - want["Gs"])
    print(K, "transitions against visits: %.1e" % (np.abs(off).max() / want["Gs"].max()))
    assert np.abs(off).max() <= 6e-8 * want["Gs"].max(), off / want["Gs"].max()
