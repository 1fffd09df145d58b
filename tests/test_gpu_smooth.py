"""Posterior probabilities, E-step statistics and gradients by strands against
the FP64 oracle, at the sizes where pieces, warm-ups and blocks of steps end,
and where vectors meet late, the recursion leaves the float range, or the
sequence is left to the chunk products.

Bar: the forward and the backward vector of a step may each be off by the
join's tolerance, 2^-15, and gamma is their normalised product: 2 x 2^-15 and
FP32 rounding, 8e-5 of the row's sum (1). The statistics are sums of such rows:
8e-5 of the largest entry of their kind.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu

STATS = ("N", "G0", "Gs", "Gr", "Sx", "Sy", "Sxx", "Sxy", "Syy")


def _check(api, prm, xy, fl, init_mode=0):
    ctx = api.Context()
    try:
        dev = api.to_device(prm)
        dxy, dfl = torch.from_numpy(np.ascontiguousarray(xy)).cuda(), torch.from_numpy(np.ascontiguousarray(fl)).cuda()
        o = api.make_opts(init_mode=init_mode)
        g, ll = ctx.hmm_posterior(*dev, dxy, dfl, opts=o)
        ref, rll = oracle.posterior(prm, xy, fl, init_mode)[:2]
        assert abs(float(ll.item()) - rll) <= 1e-6 * abs(rll) + 1e-4
        err = np.abs(g.cpu().numpy() - ref).max()
        assert err <= 8e-5, err
        if len(fl) >= 2:
            st, _ = ctx.hmm_expected_stats(*dev, dxy, dfl, opts=o)
            want = oracle.expected_stats(prm, xy, fl, init_mode)
            want = want[0] if isinstance(want, tuple) else want
            for name in STATS:
                a, b = st[name].cpu().numpy(), np.asarray(want[name])
                assert np.abs(a - b).max() <= 8e-5 * max(np.abs(b).max(), 1.0), name
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()


@pytest.mark.parametrize("K", [1, 3, 4, 7, 8, 16, 17, 25, 32, 33, 64, 65])
def test_state_counts(cuda_lib, K):
    rng = np.random.default_rng(900 + K)
    prm = synth.random_params(K, rng)
    o = synth.sample_observations(prm, 2500, rng)
    _check(cuda_lib, prm, o.xy, o.tremor)


@pytest.mark.parametrize("T", [1, 2, 3, 64, 65, 66, 67, 129, 191, 192, 193, 257, 1000, 30_001])
def test_lengths(cuda_lib, T):
    rng = np.random.default_rng(T)
    prm = synth.random_params(6, rng)
    o = synth.sample_observations(prm, T, rng)
    for init_mode in (0, 1):
        _check(cuda_lib, prm, o.xy, o.tremor, init_mode)


@pytest.mark.parametrize("K", [5, 12, 25, 40])
def test_late_meeting(cuda_lib, K):
    """Rare tremors: vectors meet after hundreds of steps, past the end of a
    piece, so that rows are written again across pieces."""
    rng = np.random.default_rng(60 + K)
    prm = synth.random_params(K, rng, p_range=synth.SPARSE_P_RANGE)
    o = synth.sample_observations(prm, 12_000, rng)
    _check(cuda_lib, prm, o.xy, o.tremor)


@pytest.mark.parametrize("K", [4, 25, 50])
def test_far_observations(cuda_lib, K):
    rng = np.random.default_rng(70 + K)
    prm = synth.random_params(K, rng)
    o = synth.sample_observations(prm, 4000, rng)
    fl, xy = o.tremor.copy(), o.xy.copy()
    at = rng.choice(4000, 40, replace=False)
    at[:2] = (0, 3999)
    fl[at] = 1
    xy[at] = rng.uniform((-300, -300), (600, 500), (40, 2)).astype(np.float32)
    _check(cuda_lib, prm, xy, fl)


def test_left_to_the_chunk_products(cuda_lib):
    """A zero in P."""
    rng = np.random.default_rng(81)
    prm = synth.random_params(6, rng)
    o = synth.sample_observations(prm, 3000, rng)
    prm.P[0, 1] += prm.P[0, 2]
    prm.P[0, 2] = 0.0
    _check(cuda_lib, prm, o.xy, o.tremor)
