"""TF32: the compensation of the vectors' truncation belongs to the steps, not
to a segment's first observation, whose vector is not truncated.

4096 segments of two observations (one step each), with a P that TF32 holds
exactly, so that the truncation of the vectors is all there is: its mean
relative loss, 3.5e-4 a step, is given back by the emissions. The random part of
a step's error is below 2^-11 / sqrt(3) = 2.8e-4, 4.4e-6 in the mean of 4096;
how far the mean loss of these vectors is from that of log-uniform mantissas is
taken as a quarter of it at most. Bar for the mean: 1e-4 a segment.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_03508_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [66, 72, 80])
def test_no_bias_by_segment(cuda_lib, K):
    api = cuda_lib
    rng = np.random.default_rng(K)
    prm = synth.random_params(K, rng)
    prm.P[:] = 1.0 / 512
    np.fill_diagonal(prm.P, (513.0 - K) / 512)
    n = 4096
    o = synth.sample_observations(prm, 2 * n, rng)
    offs = np.arange(0, 2 * n + 1, 2, dtype=np.int64)
    props = synth.stack_params([prm, prm])
    ctx = api.Context()
    try:
        got = ctx.hmm_loglik_batched(*api.to_device(props), offs, torch.from_numpy(o.xy).cuda(),
                                     torch.from_numpy(o.tremor).cuda(), opts=api.make_opts(precision="tf32")).cpu().numpy()
        assert ctx.last_chunk_proposals() == 0
        assert ctx.hmm_status() == api.HMM_OK
    finally:
        ctx.close()
    ref = oracle.loglik_batched(props, o.xy, o.tremor, offs)
    print("mean error a segment", (got - ref) / n)
    assert np.all(np.abs(got - ref) <= 1e-4 * n), (got - ref) / n
