"""Viterbi by strands against the FP64 oracle, where pieces end, where paths
coalesce late (rare tremors: pieces run again from their true vector and on
through the next), with observations far from every state, and with transition
matrices whose paths never coalesce, which the chunk products take.

Bars as in test_gpu_viterbi.py: the path's FP64 score within 1e-7 relative of
the oracle's best, the reported score within the same of the path's, and at
least 99.9% of the states equal.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


def _check(api, prm, xy, fl, mode=0):
    ctx = api.Context()
    try:
        path, score, _ = ctx.hmm_viterbi(*api.to_device(prm), torch.from_numpy(np.ascontiguousarray(xy)).cuda(),
                                         torch.from_numpy(np.ascontiguousarray(fl)).cuda(),
                                         opts=api.make_opts(init_mode=mode))
        path, score = path.cpu().numpy(), float(score.item())
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    ref_path, ref = oracle.viterbi(prm, xy, fl, mode)
    got = oracle.path_logjoint(prm, xy, fl, path, mode)
    tol = 1e-7 * abs(ref) + 1e-6
    assert got >= ref - tol, (got, ref)
    assert abs(score - got) <= tol, (score, got)
    assert np.mean(path == ref_path) >= 0.999


@pytest.mark.parametrize("K", [1, 4, 5, 9, 17, 32, 48, 64])
def test_state_counts(cuda_lib, K):
    rng = np.random.default_rng(300 + K)
    prm = synth.random_params(K, rng)
    o = synth.sample_observations(prm, 5003, rng)
    _check(cuda_lib, prm, o.xy, o.tremor)


@pytest.mark.parametrize("T", [2, 4, 127, 128, 129, 130, 257, 385, 40_001])
def test_lengths(cuda_lib, T):
    rng = np.random.default_rng(T)
    prm = synth.random_params(11, rng)
    o = synth.sample_observations(prm, T, rng)
    for mode in (0, 1):
        _check(cuda_lib, prm, o.xy, o.tremor, mode)


@pytest.mark.parametrize("K", [6, 25, 40])
def test_late_coalescence(cuda_lib, K):
    rng = np.random.default_rng(50 + K)
    prm = synth.random_params(K, rng, p_range=synth.SPARSE_P_RANGE)
    o = synth.sample_observations(prm, 20_000, rng)
    _check(cuda_lib, prm, o.xy, o.tremor)


def test_far_observations(cuda_lib):
    rng = np.random.default_rng(7)
    prm = synth.random_params(10, rng)
    o = synth.sample_observations(prm, 4000, rng)
    fl, xy = o.tremor.copy(), o.xy.copy()
    at = rng.choice(4000, 40, replace=False)
    at[:2] = (0, 3999)
    fl[at] = 1
    xy[at] = rng.uniform((-300, -300), (600, 500), (40, 2)).astype(np.float32)
    _check(cuda_lib, prm, xy, fl)


def test_paths_that_never_coalesce(cuda_lib):
    """P = I but for one pair of states, which exchange."""
    rng = np.random.default_rng(8)
    prm = synth.random_params(5, rng)
    prm.P[:] = np.eye(5, dtype=np.float32)
    prm.P[0, :2] = (0.75, 0.25)
    prm.P[1, :2] = (0.25, 0.75)
    prm.mu[:] = (150.0, 75.0) + rng.normal(0, 3, (5, 2)).astype(np.float32)
    o = synth.sample_observations(prm, 3000, rng)
    _check(cuda_lib, prm, o.xy, o.tremor)
