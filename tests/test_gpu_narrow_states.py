"""States that are narrow beside the box, strongly correlated, or far from one
another: the emissions' exponents are differences from the mean, which lose
nothing to the coordinates' size. Bars: FP32's, 1e-6 |log L| + 1e-4; 8 sqrt(T) u
as in test_gpu_tc.py for operands rounded to TF32; 8e-5 for the posterior.
"""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


def _case(K, sd, rho, away, T, seed):
    """Proposals whose means are 0.3 deviations off those the observations come from."""
    rng = np.random.default_rng(seed)
    gen = synth.random_params(K, rng)
    if away:
        gen.mu[0] = (away, away)
    gen.cov[:] = (sd * sd, rho * sd * sd, sd * sd)
    props = [synth.perturb_params(gen, rng) for _ in range(4)]
    for p in props:
        p.cov[:] = gen.cov
        p.mu[:] = gen.mu + np.float32(0.3 * sd)
    return props, synth.sample_observations(gen, T, rng)


CASES = [(0.5, 0.0, 0), (0.2, 0.0, 0), (0.05, 0.0, 0), (0.01, 0.0, 0), (0.05, 0.9, 0), (0.5, 0.99, 0), (5.0, 0.0, 1e4),
         (0.5, 0.5, 1e4)]


@pytest.mark.parametrize("sd,rho,away", CASES)
@pytest.mark.parametrize("K", [4, 25, 50])
def test_fp32(cuda_lib, K, sd, rho, away):
    api = cuda_lib
    props, o = _case(K, sd, rho, away, 30_000, K)
    xy, fl = torch.from_numpy(o.xy).cuda(), torch.from_numpy(o.tremor).cuda()
    ctx = api.Context()
    try:
        got = ctx.hmm_loglik_batched(*api.to_device(synth.stack_params(props)), [0, 30_000], xy, fl).cpu().numpy()
        g, _ = ctx.hmm_posterior(*api.to_device(props[0]), xy, fl)
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    ref = oracle.loglik_batched(synth.stack_params(props), o.xy, o.tremor, np.array([0, 30_000]), n_threads=4)
    assert np.all(np.abs(got - ref) <= 1e-6 * np.abs(ref) + 1e-4), (got - ref) / np.abs(ref)
    want, _ = oracle.posterior(props[0], o.xy, o.tremor)
    assert np.abs(g.cpu().numpy() - want).max() <= 8e-5


@pytest.mark.parametrize("sd,rho,away", CASES)
@pytest.mark.parametrize("K", [12, 28, 60])
def test_tensor_cores(cuda_lib, K, sd, rho, away):
    api = cuda_lib
    props, o = _case(K, sd, rho, away, 10_000, K)
    batch = synth.stack_params(props * 32)
    ctx = api.Context()
    try:
        got = ctx.hmm_loglik_batched(*api.to_device(batch), [0, 10_000], torch.from_numpy(o.xy).cuda(),
                                     torch.from_numpy(o.tremor).cuda(), opts=api.make_opts(precision="tf32_split")).cpu().numpy()
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    ref = oracle.loglik_batched(synth.stack_params(props), o.xy, o.tremor, np.array([0, 10_000]), n_threads=4)
    assert np.all(np.abs(got.reshape(32, 4) - ref) <= 8 * math.sqrt(10_000) * 2.0 ** -11 + 1e-3), got[:4] - ref


@pytest.mark.parametrize("K", [12, 28, 60, 80])
def test_narrow_and_ordinary_proposals_in_one_batch(cuda_lib, K):
    api = cuda_lib
    props, o = _case(K, 8.0, 0.3, 0, 10_000, K)
    for p in props[1::2]:
        p.cov[0] *= 1e-6
    batch = synth.stack_params(props * 32)
    ctx = api.Context()
    try:
        got = ctx.hmm_loglik_batched(*api.to_device(batch), [0, 4000, 10_000], torch.from_numpy(o.xy).cuda(),
                                     torch.from_numpy(o.tremor).cuda(), opts=api.make_opts(precision="tf32_split")).cpu().numpy()
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    ref = oracle.loglik_batched(synth.stack_params(props), o.xy, o.tremor, np.array([0, 4000, 10_000]), n_threads=4)
    assert np.all(np.abs(got.reshape(32, 4) - ref) <= 8 * math.sqrt(10_000) * 2.0 ** -11 + 1e-3), got[:4] - ref
