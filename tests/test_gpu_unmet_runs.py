"""Rare tremors: many pieces in a row end before their vector has met the true
one, and the rows (posterior) and back-pointers (path) they wrote from vectors
that were not the true ones have to be written again, by chains that also end
inside such pieces. Bars as in test_gpu_smooth.py (8e-5) and test_gpu_viterbi.py
(1e-7 of the best score).
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("K", [8, 14, 20, 32, 44])
def test_posterior_and_path(cuda_lib, K, seed):
    api = cuda_lib
    rng = np.random.default_rng(1500 + K + 100 * seed)
    prm = synth.random_params(K, rng, p_range=synth.SPARSE_P_RANGE)
    o = synth.sample_observations(prm, 20_000, rng)
    dev = api.to_device(prm)
    xy, fl = torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    ctx = api.Context()
    try:
        g, _ = ctx.hmm_posterior(*dev, xy, fl)
        left = ctx.last_chunk_proposals()
        path, score, _ = ctx.hmm_viterbi(*dev, xy, fl)
        print(K, seed, "left to chunk products:", left, ctx.last_chunk_proposals())
        g, path = g.cpu().numpy(), path.cpu().numpy()
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    ref, _ = oracle.posterior(prm, o.xy, o.tremor)
    assert np.abs(g - ref).max() <= 8e-5, np.abs(g - ref).max()
    _, best = oracle.viterbi(prm, o.xy, o.tremor)
    got = oracle.path_logjoint(prm, o.xy, o.tremor, path)
    assert got >= best - (1e-7 * abs(best) + 1e-6), (got, best)
    assert abs(float(score.item()) - got) <= 1e-7 * abs(best) + 1e-6
