"""Paths whose scores are close: states that emit alike and hardly exchange, told
apart by their first probabilities only. No two vectors forget that, however small
the difference; the best path stays in the likelier state. Bar as in
test_gpu_viterbi.py.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gap", [2e-2, 4e-4, 5e-5])
@pytest.mark.parametrize("K", [2, 4, 9, 20, 40])
def test_likelier_start(cuda_lib, K, gap):
    api = cuda_lib
    rng = np.random.default_rng(K)
    prm = synth.random_params(K, rng)
    prm.P[:] = 2.0 ** -20
    np.fill_diagonal(prm.P, 1.0 - (K - 1) * 2.0 ** -20)
    prm.p_tremor[:] = 0.01
    prm.pi[:] = 1.0 / K
    prm.pi[K - 1] = np.float32(math.exp(gap) / K)
    T = 1500
    xy, fl = np.zeros((T, 2), np.float32), np.zeros(T, np.uint8)
    prm.pi /= prm.pi.sum()
    ctx = api.Context()
    try:
        path, score, _ = ctx.hmm_viterbi(*api.to_device(prm), torch.from_numpy(xy).cuda(), torch.from_numpy(fl).cuda())
        path, score = path.cpu().numpy(), float(score.item())
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    _, best = oracle.viterbi(prm, xy, fl)
    got = oracle.path_logjoint(prm, xy, fl, path)
    tol = 1e-7 * abs(best) + 1e-6
    assert got >= best - tol, (got, best)
    assert abs(score - got) <= tol
