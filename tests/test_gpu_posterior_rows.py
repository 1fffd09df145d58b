"""How close the posterior's rows are where pieces meet late: each direction's
vector within its tolerance (2^-18 up to 16 states, 2^-17 up to 32, 2^-16 up to
64), once a piece; a piece's error has shrunk to half and less where the next one
ends, so four tolerances in all bound a row's two vectors: 1.5e-5, 3.1e-5, 6.1e-5
of it.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("K", [5, 9, 16, 26, 32, 48, 64])
def test_rare_tremors(cuda_lib, K, seed):
    api = cuda_lib
    rng = np.random.default_rng(40 * K + seed)
    prm = synth.random_params(K, rng, p_range=synth.SPARSE_P_RANGE)
    o = synth.sample_observations(prm, 30_000, rng)
    ctx = api.Context()
    try:
        g, _ = ctx.hmm_posterior(*api.to_device(prm), torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda())
        left = ctx.last_chunk_proposals()
        g = g.cpu().numpy()
    finally:
        ctx.close()
    ref, _ = oracle.posterior(prm, o.xy, o.tremor)
    err = float(np.abs(g - ref).max())
    print(K, seed, "error %.1e" % err, "left to chunk products:", left)
    assert err <= (1.5e-5 if K <= 16 else 3.1e-5 if K <= 32 else 6.1e-5), err
